// segsort.cu -- build every query's id list, sorted ascending.
//
// The select's traversal emits a query's ids in tree order, partly as single
// leaf hits and partly as whole subtrees (contiguous runs of the tree's id
// array).  This file gathers each query's ids from those sources and sorts
// them, with the work unit sized to the segment:
//   2..256 ids    one warp: gather into shared memory, then a bitonic network
//                 on 1-8 keys per lane in registers (shuffles across lanes,
//                 swaps inside a lane);
//   257..32256  one CTA of 64-1024 threads (16 or 32 ids each), entirely in shared
//                 memory: asynchronous copies in, buckets by value (one id
//                 each on average) counted with byte counters, and every id's
//                 rank among its bucket's neighbours gives its place in the
//                 output (cta_bucket_sort); ids in bands are bucketed again
//                 through equalized buckets, and what overflows those too
//                 (heavily repeated ids) goes to a stable LSD radix sort
//                 (8-bit digits);
//   above         cut into units for all CTAs, partitioned by value into
//                 buckets of about 8K ids through a scratch area, each bucket
//                 then sorted like a mid-size segment.
// Each class runs as a persistent grid whose CTAs claim segments from an
// atomic counter, so CTAs that drew long segments do not hold up the rest.
// LSD passes whose digit is equal for all keys are skipped (from the AND and
// OR of the keys).  In each LSD pass a key's rank among equal digits comes
// from walking the keys in order: each warp owns a contiguous run and takes it
// 32 at a time, with __match_any_sync grouping equal digits.  Keys are ids
// with the sign bit flipped, so unsigned order is signed order.
#include <climits>

#include "internal.cuh"

namespace rt {
namespace {

constexpr int kBins = 256;
constexpr int kLsdItems = 16;           // keys per thread of the LSD fallback (1024 threads); twice
                                        // that for its longest segments
constexpr int kWarpMax = 256;           // longest segment one warp sorts
constexpr uint32_t kSign = 0x80000000u;

// The ids a CTA sort takes: 252 per warp and eight ids a lane (see the
// transposition in cta_bucket_sort).
constexpr int cta_ids(int threads, int items) { return threads / 32 * (items / 8) * 252; }
constexpr int kMidMax = cta_ids(512, 32);   // longest segment below the largest class: 16128
constexpr int kCtaTop = cta_ids(1024, 32);  // longest segment of a CTA sort: 32256
static_assert(kCtaTop == kSortWhole, "the caller counts the ids that need scratch");

// Segment classes (index into the class lists).
enum {
    C_WARP = 0,  // warp sort
    C_CTA1K, C_CTA2K, C_CTA4K, C_CTA8K, C_CTA16K, C_CTA32K,  // CTA sorts
    C_LARGE,                          // split into buckets first
    C_COUNT
};
enum { HDR_SCRATCH = C_COUNT, HDR_BUCKETS, HDR_OVERSIZE, HDR_UNITS, HDR_WORDS };

struct SegDesc {
    int64_t src;  // offset of the input keys
    int64_t dst;  // offset of the output ids
    int32_t n;
    int32_t pad;
};

__device__ __forceinline__ int class_of(int64_t n)
{
    if (n <= 1) return -1;
    if (n <= kWarpMax) return C_WARP;
    if (n <= cta_ids(64, 16)) return C_CTA1K;
    if (n <= cta_ids(128, 16)) return C_CTA2K;
    if (n <= cta_ids(256, 16)) return C_CTA4K;
    if (n <= cta_ids(512, 16)) return C_CTA8K;
    if (n <= kMidMax) return C_CTA16K;
    if (n <= kCtaTop) return C_CTA32K;
    return C_LARGE;
}

// End of segment i's leaf hits in S.leaf.
__device__ __forceinline__ int64_t leaf_end(const SortSources &S, int64_t i)
{
    return S.leaf_len ? S.off_leaf[i] + S.leaf_len[i] : S.off_leaf[i + 1];
}

// Lists every segment under its class (segments of one id are written
// directly).  A block takes 256 segments at a time and reserves each class's
// list entries once: with a reservation per warp the few counters, each hit by
// every warp, took 174 us for a million segments (17 us now).
constexpr int kClassThreads = 256;
__global__ void __launch_bounds__(kClassThreads)
    k_classify(const int64_t *__restrict__ off, int64_t nseg, int32_t *__restrict__ lists, int64_t stride,
               int64_t *__restrict__ large_tmp, unsigned long long *__restrict__ hdr, SortSources S,
               int32_t *__restrict__ out, int64_t out_cap)
{
    constexpr int W = kClassThreads / 32;
    __shared__ uint32_t before[W][C_COUNT];  // entries of the warps before
    __shared__ unsigned long long base[C_COUNT];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = lanemask_lt();
    for (int64_t b = blockIdx.x * (int64_t)kClassThreads; b < nseg; b += (int64_t)gridDim.x * kClassThreads) {
        const int64_t i = b + threadIdx.x;
        int64_t len = i < nseg ? off[i + 1] - off[i] : 0;
        // a segment whose output or sources reach past a buffer's capacity is
        // skipped (the caller sees the totals exceed the capacities), and so is
        // one whose sources are not all there (the caller's flags say so)
        if (len > 0 && (off[i + 1] > out_cap || (S.left_out && S.left_out[i] < 0) ||
                        (S.leaf_cap && leaf_end(S, i) > S.leaf_cap) ||
                        (S.rng && S.rng_cap && S.off_rng[i + 1] > S.rng_cap)))
            len = 0;
        const int cls = class_of(len);
        if (len == 1) {  // a single id: copy it from its source
            int32_t v;
            if (leaf_end(S, i) > S.off_leaf[i])
                v = S.leaf[S.off_leaf[i]];
            else
                v = S.tree_ids[S.rng[S.off_rng[i]].x];
            out[off[i]] = v;
        }
        unsigned mine = 0;  // the lanes of this one's class
        for (int c = 0; c < C_COUNT; ++c) {
            const unsigned m = __ballot_sync(RT_FULL, cls == c);
            if (lane == 0)
                before[w][c] = __popc(m);
            if (cls == c)
                mine = m;
        }
        __syncthreads();
        if (threadIdx.x < C_COUNT) {
            const int c = threadIdx.x;
            uint32_t sum = 0;
            for (int x = 0; x < W; ++x) {
                const uint32_t k = before[x][c];
                before[x][c] = sum;
                sum += k;
            }
            if (sum)
                base[c] = atomicAdd(hdr + c, (unsigned long long)sum);
        }
        __syncthreads();
        if (cls >= 0) {
            const int64_t slot = (int64_t)base[cls] + before[w][cls] + __popc(mine & lt);
            lists[cls * stride + slot] = (int32_t)i;
            if (cls == C_LARGE)
                large_tmp[slot] = (int64_t)atomicAdd(hdr + HDR_SCRATCH, (unsigned long long)len);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------- gathering
// One warp copies segment i's n ids into sm[0 .. n) (in source order).
__device__ __forceinline__ void warp_gather(int32_t *__restrict__ sm, const SortSources &S,
                                            int64_t i, int n, int lane)
{
    const int64_t l0 = S.off_leaf[i], l1 = leaf_end(S, i);
    for (int64_t e = l0 + lane; e < l1; e += 32)
        sm[e - l0] = S.leaf[e];
    if (S.rng) {
        const int64_t r0 = S.off_rng[i], r1 = S.off_rng[i + 1];
        const int nl = (int)(l1 - l0);
        for (int64_t rb = r0; rb < r1; rb += 32) {
            // lanes hold up to 32 ranges, which the warp copies in turn; a
            // range ends where the next one starts
            const int64_t r = rb + lane;
            int2 rg = make_int2(0, n - nl);
            if (r < r1)
                rg = S.rng[r];
            int after = n - nl;  // the start of the range behind this chunk
            if (rb + 32 < r1)
                after = S.rng[rb + 32].y;
            const int cnt = (int)(r1 - rb < 32 ? r1 - rb : 32);
            for (int k = 0; k < cnt; ++k) {
                const int lo = __shfl_sync(RT_FULL, rg.x, k);
                const int st = __shfl_sync(RT_FULL, rg.y, k);
                const int en = k + 1 < 32 ? __shfl_sync(RT_FULL, rg.y, k + 1) : after;
                for (int e = lane; e < en - st; e += 32)
                    sm[nl + st + e] = __ldg(S.tree_ids + lo + e);
            }
        }
    }
    __syncwarp();
}

// ----------------------------------------------------------- warp sorts
// Device-resident list lengths: kernels launched without a host round trip
// read how many entries to process.
__device__ __forceinline__ int64_t list_len(const unsigned long long *count, int64_t cap)
{
    const int64_t c = (int64_t)*count;
    return c < cap ? c : cap;
}

// Bitonic sort of up to 32*K signed ids, element e = k*32 + lane (striped),
// from sm[0 .. n) to out[0 .. n).
template <int K>
__device__ __forceinline__ void warp_network(const int32_t *sm, int32_t *__restrict__ out, int n, int lane)
{
    constexpr int N = 32 * K;
    int v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = k * 32 + lane;
        v[k] = e < n ? sm[e] : INT_MAX;
    }
#pragma unroll
    for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {  // partner in the same lane, register k ^ (stride/32)
                const int ks = stride / 32;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    if (k & ks)
                        continue;
                    const int e = k * 32 + lane;
                    const bool up = (e & size) == 0;
                    const int a = v[k], b = v[k | ks];
                    v[k] = up ? min(a, b) : max(a, b);
                    v[k | ks] = up ? max(a, b) : min(a, b);
                }
            } else {  // partner in lane ^ stride, same register
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int e = k * 32 + lane;
                    const int other = __shfl_xor_sync(RT_FULL, v[k], stride);
                    const bool up = (e & size) == 0;
                    const bool lower = (lane & stride) == 0;
                    v[k] = (lower == up) ? min(v[k], other) : max(v[k], other);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = k * 32 + lane;
        if (e < n)
            out[e] = v[k];
    }
}

// Segments of 2..kWarpMax ids, one warp each.  One kernel for all lengths
// (each takes the network of its size): four kernels, most of them with little
// to do, cost a small batch four launches.
__global__ void __launch_bounds__(256) k_sort_warp(const int32_t *__restrict__ list,
                                                   const unsigned long long *__restrict__ count,
                                                   int64_t cap, const int64_t *__restrict__ off,
                                                   SortSources S, int32_t *__restrict__ out)
{
    const int64_t cnt = list_len(count, cap);
    __shared__ int32_t stage[8][kWarpMax];
    const int lane = threadIdx.x & 31;
    int32_t *sm = stage[threadIdx.x >> 5];
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t wi = warp; wi < cnt; wi += nwarps) {
        const int32_t seg = list[wi];
        const int64_t o = off[seg];
        const int n = (int)(off[seg + 1] - o);
        warp_gather(sm, S, seg, n, lane);
        if (n <= 32)
            warp_network<1>(sm, out + o, n, lane);
        else if (n <= 64)
            warp_network<2>(sm, out + o, n, lane);
        else if (n <= 128)
            warp_network<4>(sm, out + o, n, lane);
        else
            warp_network<8>(sm, out + o, n, lane);
        __syncwarp();
    }
}

// ------------------------------------------------------------ CTA sort
constexpr int kHalo = 32;          // slots kept before and after the keys (a window is at most 31)
constexpr int kNet = 5;            // ids a bucket may hold for the register network
constexpr int kCoarse = 4;         // coarse bins per thread of the equalized buckets
constexpr int kRetry = 12;         // a bucket this full asks for equalized buckets
constexpr int kLongRange = 2048;   // longer id runs are copied by the whole CTA

// A segment to sort: n ids of which nl are leaf hits, nr whole subtrees.
struct Piece {
    int64_t dst;  // where its ids go in the output
    int64_t src;  // its leaf hits in S.leaf (or its ids in the scratch area)
    int64_t rng;  // its ranges in S.rng
    int32_t n;    // < 0: nothing left
    int32_t nl;
    int32_t nr;
    int32_t seg;  // list entry: the segment
};

// Shared memory of one CTA sort: 4 bytes of key and 1 byte of bucket counter
// per id.
template <int THREADS, int ITEMS>
struct CtaSmem {
    static constexpr int N = cta_ids(THREADS, ITEMS);
    static_assert(ITEMS % 16 == 0 && THREADS % 32 == 0, "a thread's counter words are read 16 bytes at a time");
    uint32_t slots[THREADS * ITEMS + 192];  // kHalo smallest ids, then the ids and their upper halo
    uint32_t cnt[THREADS * ITEMS / 4];       // four byte counters a word; then the packed bucket starts
    uint32_t win[THREADS * ITEMS / 32 + 4];       // per 32 positions: largest bucket of more than kNet there, less one
    uint32_t coarse[kCoarse * THREADS + 2];  // equalized buckets: first bucket of each coarse bin
    uint32_t red0[32], red1[32];       // per-warp partial results
    Piece next;                        // the segment this CTA takes next
    __device__ __forceinline__ uint32_t *buf() { return slots + kHalo; }
};

// Exclusive block scan of one int per thread (w: one word per warp); returns
// the prefix and writes the block total to *total.  One barrier: the caller
// has another before w is written again.
template <int THREADS>
__device__ __forceinline__ int block_scan_int(uint32_t *w, int v, int *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(RT_FULL, inc, o);
        if (lane >= o)
            inc += u;
    }
    if (lane == 31)
        w[wid] = (uint32_t)inc;
    __syncthreads();
    const unsigned s = lane < THREADS / 32 ? w[lane] : 0u;
    *total = (int)__reduce_add_sync(RT_FULL, s);
    return (int)__reduce_add_sync(RT_FULL, lane < wid ? s : 0u) + inc - v;
}

// Block-wide minimum and maximum (w0, w1: one word per warp); every thread
// gets both.  One barrier, as block_scan_int.
template <int THREADS>
__device__ __forceinline__ void block_minmax(uint32_t *w0, uint32_t *w1, int &kmin, int &kmax)
{
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    kmin = __reduce_min_sync(RT_FULL, kmin);
    kmax = __reduce_max_sync(RT_FULL, kmax);
    if (lane == 0) {
        w0[wid] = (uint32_t)kmin;
        w1[wid] = (uint32_t)kmax;
    }
    __syncthreads();
    kmin = __reduce_min_sync(RT_FULL, lane < THREADS / 32 ? (int)w0[lane] : INT_MAX);
    kmax = __reduce_max_sync(RT_FULL, lane < THREADS / 32 ? (int)w1[lane] : INT_MIN);
}

__device__ __forceinline__ void cp_async4(uint32_t *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// `lanes` threads (this one is number t) start the copy of src[0 .. n) into
// shared memory: 16 bytes at a time where both sides are aligned.
__device__ __forceinline__ void copy_async(uint32_t *dst, const int32_t *src, int n, int t, int lanes)
{
    const unsigned both = (unsigned)(uintptr_t)src | (unsigned)__cvta_generic_to_shared(dst);
    int done = 0;
    if ((both & 15u) == 0) {
        done = n & ~3;
        for (int e = 4 * t; e < done; e += 4 * lanes)
            cp_async16(dst + e, src + e);
    }
    for (int e = done + t; e < n; e += lanes)
        cp_async4(dst + e, src + e);
}

// The CTA starts copying piece m's ids into shared memory: the ids of its
// whole subtrees first, then its leaf hits.  The copies are asynchronous
// (cp.async), so every range's loads are in flight together: with a register
// copy each warp waited for one range at a time, which was a third of the
// sort's time.  Subtree runs of full leaves keep 16-byte alignment on both
// sides, and so do leaf hits in slots reserved F at a time.
template <int THREADS, int ITEMS>
__device__ __forceinline__ void cta_gather(CtaSmem<THREADS, ITEMS> &sm, const SortSources &S, const Piece &m)
{
    uint32_t *buf = sm.buf();
    const int nrl = m.n - m.nl;
    copy_async(buf + nrl, S.leaf + m.src, m.nl, threadIdx.x, THREADS);
    // 4 to 32 lanes a range: 16 bytes a lane copy the average one
    const int lg = nrl > 64 * m.nr ? 5 : nrl > 32 * m.nr ? 4 : nrl > 16 * m.nr ? 3 : 2;
    const int sub = threadIdx.x & ((1 << lg) - 1);
    const int2 *rng = S.rng + m.rng;
    bool some_long = false;
    for (int k = threadIdx.x >> lg; k < m.nr; k += THREADS >> lg) {
        const int2 g = rng[k];
        const int e = k + 1 < m.nr ? rng[k + 1].y : nrl;
        if (e - g.y > kLongRange)
            some_long = true;
        else if (g.y >= 0 && e <= nrl)
            copy_async(buf + g.y, S.tree_ids + g.x, e - g.y, sub, 1 << lg);
    }
    if (__syncthreads_or(some_long)) {  // longer ranges: the whole CTA, one after another
        for (int b = 0; b < m.nr; b += 32) {
            const int k = b + (int)(threadIdx.x & 31);
            int2 g = make_int2(0, 0);
            int e = 0;
            if (k < m.nr) {
                g = rng[k];
                e = k + 1 < m.nr ? rng[k + 1].y : nrl;
            }
            unsigned todo = __ballot_sync(RT_FULL, e - g.y > kLongRange && g.y >= 0 && e <= nrl);
            while (todo) {
                const int l = __ffs(todo) - 1;
                todo &= todo - 1;
                const int lo = __shfl_sync(RT_FULL, g.x, l), st = __shfl_sync(RT_FULL, g.y, l);
                const int en = __shfl_sync(RT_FULL, e, l);
                copy_async(buf + st, S.tree_ids + lo, en - st, threadIdx.x, THREADS);
            }
        }
    }
}

// Value buckets: id * mult + add as a 64-bit product is (id - smallest id) *
// mult; its high word is the bucket (one multiply-add an id).
// Plain: n equal parts of the id range.  Equalized: kCoarse * THREADS equal coarse
// bins of the range, each cut into as many equal parts as it holds ids (the
// product's low word is the place within the bin).  Both are monotone.
struct BucketMap {
    int mult;
    int64_t add;
    const uint32_t *coarse;
};
__device__ __forceinline__ uint32_t coarse_of(const BucketMap &m, int id)
{
    return (uint32_t)(((int64_t)id * m.mult + m.add) >> 32);
}
template <bool EQ>
__device__ __forceinline__ uint32_t bucket_of(const BucketMap &m, int id)
{
    if (!EQ)
        return coarse_of(m, id);
    const uint64_t p = (uint64_t)((int64_t)id * m.mult + m.add);
    const uint32_t c = (uint32_t)(p >> 32);
    const uint32_t h0 = m.coarse[c];
    return h0 + __umulhi((uint32_t)p, m.coarse[c + 1] - h0);
}
// mult = parts * 2^32 / (range + 1), rounded down past float's rounding error
// so that the largest id maps below `parts` (and below 2^31: a range shorter
// than 2 * parts then leaves the upper parts empty).
__device__ __forceinline__ BucketMap bucket_map(int parts, int kmin, int kmax, const uint32_t *coarse)
{
    const float span = (float)((uint32_t)kmax - (uint32_t)kmin);
    const float m = (float)parts * 4294967296.f / (span + 1.f) * (1.f - 4.76837158e-7f);
    BucketMap b;
    b.mult = m < 2147483520.f ? (int)m : 2147483520;
    b.add = -(int64_t)kmin * b.mult;
    b.coarse = coarse;
    return b;
}

// Calls f(k, p) for each of the thread's keys: key k of the thread is element
// p = 4*THREADS*(k/4) + 4*threadIdx.x + k%4 of the n.  Whole rounds of
// 4*THREADS elements need no test per key; only the last one tests (a branch
// per key was a fifth of the instructions).
template <int THREADS, int ITEMS, typename F>
__device__ __forceinline__ void each_key(int n, F f)
{
    const int p0 = (int)threadIdx.x * 4;
#pragma unroll
    for (int i = 0; i < ITEMS / 4; ++i) {
        if ((i + 1) * 4 * THREADS <= n) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                f(4 * i + j, i * 4 * THREADS + p0 + j);
        } else if (i * 4 * THREADS < n) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i * 4 * THREADS + p0 + j < n)
                    f(4 * i + j, i * 4 * THREADS + p0 + j);
        }
    }
}

// Counts the keys into byte counters (each key's arrival number within its
// bucket stays in `arr`), and turns the counters into bucket starts, packed
// {start of the word's first bucket: 17 bits; keys before its fourth, third
// and second bucket: 5 bits each}.  Needs cnt and win zeroed.  False if a
// field overflowed (the starts are unusable) or, for plain buckets, if one
// holds kRetry keys or more.
template <int THREADS, int ITEMS, bool EQ>
__device__ __forceinline__ bool count_buckets(CtaSmem<THREADS, ITEMS> &sm, const BucketMap &bm,
                                              const int (&key)[ITEMS], uint32_t (&arr)[ITEMS / 4], int n)
{
    constexpr int WORDS = ITEMS / 4;  // counter words of a thread
    each_key<THREADS, ITEMS>(n, [&](int k, int) {
        const uint32_t b = bucket_of<EQ>(bm, key[k]);
        const uint32_t sh = (b << 3) & 31u;
        const uint32_t old = atomicAdd(&sm.cnt[b >> 2], 1u << sh);
        const uint32_t a = old >> sh;  // its low byte goes to byte k%4
        const int j = k & 3;
        arr[k >> 2] = j == 0 ? a : __byte_perm(arr[k >> 2], a, j == 1 ? 0x3240 : j == 2 ? 0x3410 : 0x4210);
    });
    __syncthreads();
    const int w0 = (int)threadIdx.x * WORDS;
    const bool mine = w0 < ((n + 3) >> 2);
    uint32_t w[WORDS], over = 0, top = 0, sum = 0;
    if (mine) {
#pragma unroll
        for (int k = 0; k < WORDS; k += 4) {
            const uint4 a = *reinterpret_cast<const uint4 *>(sm.cnt + w0 + k);
            w[k] = a.x, w[k + 1] = a.y, w[k + 2] = a.z, w[k + 3] = a.w;
        }
#pragma unroll
        for (int k = 0; k < WORDS; ++k) {
            over |= w[k] & 0xe0e0e0e0u;
            top = __vmaxu2(top, __vmaxu2(w[k] & 0x00ff00ffu, (w[k] >> 8) & 0x00ff00ffu));
            sum = __dp4a(w[k], 0x01010101u, sum);
        }
    }
    // a counter past 255 carries into the next one or out of the word, which
    // only ever makes the total smaller than n
    int total;
    uint32_t run = (uint32_t)block_scan_int<THREADS>(sm.red0, (int)sum, &total);
    const uint32_t biggest = max(top & 0xffffu, top >> 16);
    if (mine) {
        if (biggest > (uint32_t)kNet && total == n)
            for (uint32_t c = run >> 5; c <= (run + sum - 1) >> 5; ++c)
                atomicMax(&sm.win[c], biggest - 1);
#pragma unroll
        for (int k = 0; k < WORDS; ++k) {
            const uint32_t pre = w[k] * 0x01010100u;  // byte q: keys before the word's bucket q
            const uint32_t next = run + (pre >> 24) + (w[k] >> 24);
            over |= pre & 0xe0e0e000u;
            w[k] = (run << 15) | ((pre >> 8) & 31u) | ((pre >> 11) & (31u << 5)) | ((pre >> 14) & (31u << 10));
            run = next;
        }
#pragma unroll
        for (int k = 0; k < WORDS; k += 4)
            *reinterpret_cast<uint4 *>(sm.cnt + w0 + k) = make_uint4(w[k], w[k + 1], w[k + 2], w[k + 3]);
    }
    return __syncthreads_or(over != 0 || total != n || (!EQ && biggest >= (uint32_t)kRetry)) == 0;
}

// Moves the keys (all of them in registers) to their buckets in sm.buf().
template <int THREADS, int ITEMS, bool EQ>
__device__ __forceinline__ void scatter_buckets(CtaSmem<THREADS, ITEMS> &sm, const BucketMap &bm,
                                                const int (&key)[ITEMS], const uint32_t (&arr)[ITEMS / 4], int n)
{
    uint32_t *buf = sm.buf();
    each_key<THREADS, ITEMS>(n, [&](int k, int) {
        const uint32_t b = bucket_of<EQ>(bm, key[k]);
        const uint32_t v = sm.cnt[b >> 2];
        buf[(v >> 15) + (((v << 5) >> (5 * (b & 3u))) & 31u) + __byte_perm(arr[k >> 2], 0, 0x4440 | (k & 3))] = (uint32_t)key[k];
    });
}

template <int THREADS, int ITEMS>
__device__ __forceinline__ void zero_counters(CtaSmem<THREADS, ITEMS> &sm, int n)
{
    uint4 *c = reinterpret_cast<uint4 *>(sm.cnt);
    const int n4 = ((n + 31) >> 5) * 2;  // whole groups of 8 words (32 buckets)
    for (int k = threadIdx.x; k < n4; k += THREADS)
        c[k] = make_uint4(0, 0, 0, 0);
    for (int k = threadIdx.x; k < (n >> 5) + 4; k += THREADS)
        sm.win[k] = 0;
}

// Sorts the n ids in sm.buf() and writes them to dst.
//
// The ids are bucketed by value, one bucket per id on average.  After the
// scatter into bucket order an id is at most (its bucket's size - 1) places
// from where it belongs, so a few rounds of odd-even transposition finish the
// sort: kNet rounds in registers sort every bucket of up to kNet ids, and
// where a larger one lies (win) the write-out counts inversions instead: an
// id at p belongs at p + (later ids smaller than it) - (earlier ids larger).
//
// Bound by shared memory and by instruction issue together, in phases that
// barriers separate (22 to 24 wavefronts and 94 to 118 warp instructions per 32
// ids, 27 and 130 in the smallest class: about half of the peak of either; the
// random atomics, loads and stores of the count and the scatter are ten of the 22).
// All classes on 1.43G ids (10M rectangles, 1M queries): 7.65 ms, against
// 10.4 ms with buckets of three to five ids sorted by per-thread bitonic
// networks, a third of whose instructions were the networks' padding.
//
// Ids that fill some buckets with kRetry or more (ids in bands, e.g. rows
// stored region by region) are bucketed again through equalized buckets.  If
// those overflow too (heavily repeated ids) the function returns false with
// the unsorted ids in dst, and the caller sorts them another way.
// after_count and before_write are called on the way, by all threads (unless
// the function returns early): the caller's loads for the next piece.
template <int THREADS, int ITEMS, typename P1, typename P2>
__device__ __forceinline__ bool cta_bucket_sort(CtaSmem<THREADS, ITEMS> &sm, int32_t *__restrict__ dst, int n,
                                                P1 after_count, P2 before_write)
{
    uint32_t *buf = sm.buf();
    const int lane = threadIdx.x & 31;
    int key[ITEMS];
    uint32_t arr[ITEMS / 4];
    int kmin = INT_MAX, kmax = INT_MIN;
#pragma unroll
    for (int i = 0; i < ITEMS / 4; ++i) {
        if (i * 4 * THREADS < n) {
            const int4 v = *reinterpret_cast<const int4 *>(buf + (i * THREADS + threadIdx.x) * 4);
            key[4 * i] = v.x, key[4 * i + 1] = v.y, key[4 * i + 2] = v.z, key[4 * i + 3] = v.w;
            if ((i + 1) * 4 * THREADS <= n) {
                kmin = __vimin3_s32(kmin, __vimin3_s32(v.x, v.y, v.z), v.w);
                kmax = __vimax3_s32(kmax, __vimax3_s32(v.x, v.y, v.z), v.w);
            } else {
                const int p = (i * THREADS + (int)threadIdx.x) * 4;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (p + j < n) {
                        kmin = min(kmin, key[4 * i + j]);
                        kmax = max(kmax, key[4 * i + j]);
                    }
                }
            }
        }
    }
    block_minmax<THREADS>(sm.red0, sm.red1, kmin, kmax);
    if (kmin == kmax) {  // all ids equal
        for (int p = threadIdx.x; p < n; p += THREADS)
            dst[p] = kmin;
        return true;
    }
    BucketMap bm = bucket_map(n, kmin, kmax, sm.coarse);
    bool eq = false;
    if (!count_buckets<THREADS, ITEMS, false>(sm, bm, key, arr, n)) {
        eq = true;
        constexpr int C = kCoarse * THREADS;  // coarse bins
        bm = bucket_map(C, kmin, kmax, sm.coarse);
        zero_counters(sm, n);
#pragma unroll
        for (int k = 0; k < kCoarse; ++k)
            sm.coarse[k * THREADS + threadIdx.x] = 0;
        __syncthreads();
        each_key<THREADS, ITEMS>(n, [&](int k, int) { atomicAdd(&sm.coarse[coarse_of(bm, key[k])], 1u); });
        __syncthreads();
        uint32_t h[kCoarse], sum = 0;
#pragma unroll
        for (int k = 0; k < kCoarse; ++k) {
            h[k] = sm.coarse[kCoarse * threadIdx.x + k];
            sum += h[k];
        }
        int total;
        uint32_t run = (uint32_t)block_scan_int<THREADS>(sm.red1, (int)sum, &total);
#pragma unroll
        for (int k = 0; k < kCoarse; ++k) {
            sm.coarse[kCoarse * threadIdx.x + k] = run;
            run += h[k];
        }
        if (threadIdx.x == 0)
            sm.coarse[C] = (uint32_t)total;
        __syncthreads();
        if (!count_buckets<THREADS, ITEMS, true>(sm, bm, key, arr, n)) {
            each_key<THREADS, ITEMS>(n, [&](int k, int p) { dst[p] = key[k]; });
            return false;
        }
    }
    after_count();
    if (threadIdx.x < kHalo)
        buf[n + threadIdx.x] = (uint32_t)INT_MAX;
    if (eq)
        scatter_buckets<THREADS, ITEMS, true>(sm, bm, key, arr, n);
    else
        scatter_buckets<THREADS, ITEMS, false>(sm, bm, key, arr, n);
    __syncthreads();
    // Eight consecutive positions a thread and round, with four neighbours on
    // either side: five rounds of odd-even transposition over the whole array
    // (each thread computes what its own eight depend on).  A warp's tile is
    // 252 positions: the lanes with bit 2 set start 124 positions on, so that
    // the eight lanes of one 128-byte access phase hit different banks (the
    // four positions both halves compute are equal).
    const int place = (lane & 4) * 31 + 8 * ((lane & 3) | (lane >> 3 << 2));
#pragma unroll
    for (int i = 0; i < ITEMS / 8; ++i) {
        const int p = (i * (THREADS / 32) + (int)(threadIdx.x >> 5)) * 252 + place;
        if (p < n) {
            int v[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int4 x = *reinterpret_cast<const int4 *>(buf + p - 4 + 4 * q);
                v[4 * q] = x.x, v[4 * q + 1] = x.y, v[4 * q + 2] = x.z, v[4 * q + 3] = x.w;
            }
#pragma unroll
            for (int r = 0; r < kNet; ++r) {
#pragma unroll
                for (int j = r; j < 15 - r; j += 2) {
                    const int lo = min(v[j], v[j + 1]), hi = max(v[j], v[j + 1]);
                    v[j] = lo;
                    v[j + 1] = hi;
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                key[8 * i + j] = v[4 + j];
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS / 8; ++i) {
        const int p = (i * (THREADS / 32) + (int)(threadIdx.x >> 5)) * 252 + place;
        if (p < n) {
            *reinterpret_cast<int4 *>(buf + p) = make_int4(key[8 * i], key[8 * i + 1], key[8 * i + 2], key[8 * i + 3]);
            *reinterpret_cast<int4 *>(buf + p + 4) =
                make_int4(key[8 * i + 4], key[8 * i + 5], key[8 * i + 6], key[8 * i + 7]);
        }
    }
    __syncthreads();
    before_write();
    // write-out, a warp 128 positions at a time
    for (int p0 = (threadIdx.x >> 5) * 128; p0 < n; p0 += 4 * THREADS) {
        const int *at = reinterpret_cast<const int *>(buf) + p0 + lane;
        int32_t *to = dst + p0 + lane;
        const uint4 w = *reinterpret_cast<const uint4 *>(sm.win + (p0 >> 5));
        int k[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            k[u] = at[32 * u];
        if (p0 + 128 <= n && (w.x | w.y | w.z | w.w) == 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                to[32 * u] = k[u];
        } else {  // the end of the segment, or a bucket too large for the network: count inversions
            const int widest = (int)max(max(w.x, w.y), max(w.z, w.w));
            int move[4] = {0, 0, 0, 0};
            for (int d = 1; d <= widest; ++d) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    move[u] += at[32 * u + d] < k[u];
                    move[u] -= at[32 * u - d] > k[u];
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (p0 + 32 * u + lane < n)
                    to[32 * u + move[u]] = k[u];
        }
    }
    return true;
}

__device__ __forceinline__ void push_crowded(SegDesc *list, unsigned long long *count, int64_t cap,
                                             int64_t dst, int n)
{
    const unsigned long long slot = atomicAdd(count, 1ull);
    if ((int64_t)slot < cap)
        list[slot] = SegDesc{dst, dst, n, 0};
}

constexpr int cta_per_sm(int threads, int items) { return (items <= 16 ? 1536 : 1024) / threads; }

// One CTA per listed segment.  BUCKETS: the list holds SegDesc entries whose
// ids sit in `scratch`; otherwise segment ids whose ids are gathered from S.
// CTAs claim list entries from the counter *next (zero at launch), so
// a CTA that drew short segments takes more.
template <int THREADS, int ITEMS, bool BUCKETS>
__global__ void __launch_bounds__(THREADS, cta_per_sm(THREADS, ITEMS))
    k_sort_cta(const void *__restrict__ list, const unsigned long long *__restrict__ count,
               int64_t list_cap, const int64_t *__restrict__ off, SortSources S,
               const int32_t *__restrict__ scratch, int32_t *__restrict__ out,
               SegDesc *__restrict__ crowded, unsigned long long *__restrict__ n_crowded,
               int64_t crowded_cap, unsigned long long *__restrict__ next)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using Smem = CtaSmem<THREADS, ITEMS>;
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int64_t cnt = list_len(count, list_cap);
    if (threadIdx.x < kHalo)
        sm.slots[threadIdx.x] = (uint32_t)INT_MIN;
    // The next piece is claimed and its description loaded by the first warp
    // while the current one is sorted, one dependent load per phase (claim,
    // list entry, offsets); the chain's latency was a tenth of the time of
    // the largest class, of which an SM holds one CTA.
    const bool first = threadIdx.x < 32;
    unsigned long long claimed = 0;
    int32_t seg = -1;
    int64_t v = 0;
    int32_t hits = 0;
    auto claim = [&] {
        if (threadIdx.x == 0)
            claimed = atomicAdd(next, 1ull);
    };
    auto load_entry_of_list = [&] {
        if (!first)
            return;
        const long long c = (long long)__shfl_sync(RT_FULL, claimed, 0);
        seg = c >= cnt ? -1 : BUCKETS ? (int32_t)c : static_cast<const int32_t *>(list)[c];
    };
    auto load_fields = [&] {  // lane j: field j
        const int j = threadIdx.x;
        v = 0;
        if (!first || seg < 0)
            return;
        if (BUCKETS) {
            const SegDesc *d = static_cast<const SegDesc *>(list) + seg;
            v = j == 0 ? d->dst : j == 1 ? d->n : j == 2 ? d->src : 0;
        } else {
            const int64_t *at = j < 2 ? off + seg + j : j < 4 ? S.off_leaf + seg + (j - 2) : S.off_rng + seg + (j - 4);
            if (j < 4 || (j < 6 && S.rng))
                v = *at;
            hits = S.leaf_len ? S.leaf_len[seg] : 0;
        }
    };
    auto store_piece = [&] {
        if (!first)
            return;
        const int64_t f0 = __shfl_sync(RT_FULL, v, 0), f1 = __shfl_sync(RT_FULL, v, 1), f2 = __shfl_sync(RT_FULL, v, 2),
                      f3 = __shfl_sync(RT_FULL, v, 3), f4 = __shfl_sync(RT_FULL, v, 4), f5 = __shfl_sync(RT_FULL, v, 5);
        if (threadIdx.x == 0) {
            Piece m;
            m.dst = f0;
            m.src = f2;
            m.rng = f4;
            m.n = seg < 0 ? -1 : (int)(BUCKETS ? f1 : f1 - f0);
            const int64_t nl = BUCKETS ? f1 : S.leaf_len ? hits : f3 - f2;
            m.nl = (int)(nl < m.n ? nl : m.n);
            m.nr = (int)(f5 - f4);
            m.seg = seg;
            sm.next = m;
        }
    };
    claim();
    load_entry_of_list();
    load_fields();
    store_piece();
    for (;;) {
        __syncthreads();  // also: the previous piece is done with the shared memory
        const Piece m = sm.next;
        if (m.n < 0)
            break;
        claim();
        bool ok = true;
        bool loaded = false;
        if (m.n <= Smem::N) {
            zero_counters(sm, m.n);
            if (BUCKETS)
                copy_async(sm.buf(), scratch + m.src, m.n, threadIdx.x, THREADS);
            else
                cta_gather(sm, S, m);
            cp_async_wait();
            __syncthreads();
            ok = cta_bucket_sort(sm, out + m.dst, m.n, load_entry_of_list, [&] {
                load_fields();
                loaded = true;
            });
        } else {
            __syncthreads();  // every thread has read sm.next
        }
        if (!loaded) {
            load_entry_of_list();
            load_fields();
        }
        store_piece();
        if (!ok && threadIdx.x == 0)
            push_crowded(crowded, n_crowded, crowded_cap, m.dst, m.n);
    }
}

// Shared memory of the LSD fallback.
template <int ITEMS>
struct LsdSmem {
    static constexpr int W = 32;
    uint32_t buf[1024 * ITEMS];
    uint32_t wcnt[W][kBins];
    uint32_t dcount[kBins];
    uint32_t dstart[kBins];
    uint32_t red0[W], red1[W];
};

// Block-wide AND and OR of the keys' bits; every thread gets AND ^ OR.
template <int ITEMS>
__device__ __forceinline__ uint32_t block_diff(LsdSmem<ITEMS> &sm, uint32_t a_and, uint32_t a_or)
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    a_and = __reduce_and_sync(RT_FULL, a_and);
    a_or = __reduce_or_sync(RT_FULL, a_or);
    if (lane == 0) {
        sm.red0[w] = a_and;
        sm.red1[w] = a_or;
    }
    __syncthreads();
    a_and = __reduce_and_sync(RT_FULL, sm.red0[lane]);
    a_or = __reduce_or_sync(RT_FULL, sm.red1[lane]);
    __syncthreads();
    return a_and ^ a_or;
}

// Ranks the keys held in registers for one LSD pass; on return pos[i] is the
// position of key[i] in the pass's output order.  Warp w owns keys
// [w*run, (w+1)*run), taken 32 at a time.
template <int THREADS, int ITEMS>
__device__ __forceinline__ void rank_pass(LsdSmem<ITEMS> &sm, const uint32_t (&key)[ITEMS],
                                          int rounds, int run, int n, int shift,
                                          uint32_t (&pos)[ITEMS])
{
    constexpr int W = THREADS / 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    for (int i = threadIdx.x; i < W * kBins; i += THREADS)
        (&sm.wcnt[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if (i >= rounds)
            break;
        const bool ok = w * run + i * 32 + lane < n;
        const int dg = ok ? (int)((key[i] >> shift) & 0xffu) : kBins;
        const unsigned peers = __match_any_sync(RT_FULL, dg);
        const uint32_t prev = ok ? sm.wcnt[w][dg] : 0u;
        pos[i] = prev + __popc(peers & lt);
        __syncwarp();
        if (ok && lane == __ffs(peers) - 1)
            sm.wcnt[w][dg] = prev + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kBins; d += THREADS) {
        uint32_t r = 0;
#pragma unroll 8
        for (int x = 0; x < W; ++x) {
            const uint32_t c = sm.wcnt[x][d];
            sm.wcnt[x][d] = r;
            r += c;
        }
        sm.dcount[d] = r;
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // exclusive scan of the 256 digit totals by one warp
        uint32_t carry = 0;
#pragma unroll
        for (int c = 0; c < kBins; c += 32) {
            const uint32_t v = sm.dcount[c + lane];
            uint32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(RT_FULL, inc, o);
                if (lane >= o)
                    inc += u;
            }
            sm.dstart[c + lane] = carry + inc - v;
            carry += __shfl_sync(RT_FULL, inc, 31);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if (i >= rounds)
            break;
        if (w * run + i * 32 + lane < n) {
            const int dg = (int)((key[i] >> shift) & 0xffu);
            pos[i] += sm.dstart[dg] + sm.wcnt[w][dg];
        }
    }
}

// Stable LSD radix sort of n <= 1024 * ITEMS ids in place at ids[0 .. n).
template <int ITEMS>
__device__ __forceinline__ void cta_lsd_sort(LsdSmem<ITEMS> &sm, int32_t *__restrict__ ids, int n)
{
    constexpr int THREADS = 1024, W = 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int run = ((n + W * 32 - 1) / (W * 32)) * 32;
    const int rounds = run / 32;
    uint32_t key[ITEMS], pos[ITEMS];
    uint32_t a_and = 0xffffffffu, a_or = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        key[i] = 0;
        const int p = w * run + i * 32 + lane;
        if (i < rounds && p < n) {
            key[i] = (uint32_t)ids[p] ^ kSign;
            a_and &= key[i];
            a_or |= key[i];
        }
    }
    const uint32_t diff = block_diff(sm, a_and, a_or);
    int last = -1;
    for (int shift = 0; shift < 32; shift += 8)
        if ((diff >> shift) & 0xffu)
            last = shift;
    for (int shift = 0; shift <= last; shift += 8) {
        if (((diff >> shift) & 0xffu) == 0)
            continue;
        rank_pass<THREADS, ITEMS>(sm, key, rounds, run, n, shift, pos);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (i < rounds && w * run + i * 32 + lane < n)
                sm.buf[pos[i]] = key[i];
        __syncthreads();
        if (shift == last) {
            for (int p = threadIdx.x; p < n; p += THREADS)
                ids[p] = (int32_t)(sm.buf[p] ^ kSign);
        } else {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int p = w * run + i * 32 + lane;
                if (i < rounds && p < n)
                    key[i] = sm.buf[p];
            }
        }
        __syncthreads();
    }
}

// Segments whose buckets were crowded, sorted in place by LSD radix: those of
// least .. 1024 * ITEMS ids.  Persistent: the list length is read on the device.
template <int ITEMS>
__global__ void __launch_bounds__(1024, 1)
    k_sort_lsd(const SegDesc *__restrict__ list, const unsigned long long *__restrict__ count,
               int64_t cap, int least, int32_t *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LsdSmem<ITEMS> &sm = *reinterpret_cast<LsdSmem<ITEMS> *>(smem_raw);
    const int64_t cnt = list_len(count, cap);
    for (int64_t b = blockIdx.x; b < cnt; b += gridDim.x) {
        const SegDesc d = list[b];
        if (d.n >= least && d.n <= 1024 * ITEMS)
            cta_lsd_sort(sm, out + d.dst, d.n);
    }
}

// ------------------------------------------------------------ long segments
// A segment too long for a CTA sort is cut into units of kUnit ids that any CTA can
// take (with a CTA per segment a batch of a few dozen windows left most SMs
// idle), and partitioned by value into buckets a CTA sort takes:
//   k_long_plan     per segment: the ids' range from a sample, its units;
//   k_long_gather   per unit: ids into their place in the output (unsorted),
//                   and counted into the segment's kBinsLong value bins;
//   k_long_split    per segment: consecutive bins become buckets of about
//                   kBucketIds ids, listed for the CTA sort;
//   k_long_scatter  per unit: ids to their buckets in the scratch area.
// Ids outside the sample's range go to the end bins.
// 40 windows of 185K ids on average: 200 us for their whole sort, 630 us with
// one CTA a segment for the gather and the partition; a plan batch with 800
// such windows among 100K queries: 2.26 ms, before 2.66.
// 4096 ids a unit: its CTA (21 or 31 KB of shared memory) fits beside the
// persistent CTAs of the large sort classes, which leave 41 KB of an SM; units
// of 8192 waited for those to finish and ended the sort late.
constexpr int kUnit = 4096;
constexpr int kBinsLong = 1024;
constexpr int kBucketIds = 8192;
constexpr int kSample = 2048;

struct LongSeg {
    int64_t add;     // value map: bin = (id * mult + add) >> 32, clamped
    int32_t mult;
    int32_t pad;
};
struct Unit {
    int32_t slot;  // in the long segments' list
    int32_t part;  // which kUnit ids of it
};

__device__ __forceinline__ int bin_of(const LongSeg &g, int id)
{
    const int b = (int)(((int64_t)id * g.mult + g.add) >> 32);
    return max(0, min(kBinsLong - 1, b));
}

__global__ void __launch_bounds__(256)
    k_long_plan(const int32_t *__restrict__ list, const unsigned long long *__restrict__ count, int64_t list_cap,
                const int64_t *__restrict__ tmp_off, int64_t scratch_cap, const int64_t *__restrict__ off,
                SortSources S, LongSeg *__restrict__ segs, uint32_t *__restrict__ hist, Unit *__restrict__ units,
                int64_t unit_cap, unsigned long long *__restrict__ hdr, int32_t *__restrict__ flags)
{
    __shared__ int red[2][8];
    __shared__ unsigned long long first;
    const int64_t cnt = list_len(count, list_cap);
    for (int64_t b = blockIdx.x; b < cnt; b += gridDim.x) {
        const int32_t i = list[b];
        const int64_t n = off[i + 1] - off[i];
        const int64_t l0 = S.off_leaf[i], nl = leaf_end(S, i) - l0;
        const int64_t r0 = S.rng ? S.off_rng[i] : 0, nr = S.rng ? S.off_rng[i + 1] - r0 : 0;
        int lo = INT_MAX, hi = INT_MIN;
        for (int k = threadIdx.x; k < kSample; k += 256) {
            if (nr > 0) {  // an id of every few runs
                const int v = S.tree_ids[S.rng[r0 + nr * k / kSample].x];
                lo = min(lo, v), hi = max(hi, v);
            }
            if (nl > 0) {
                const int v = S.leaf[l0 + nl * k / kSample];
                lo = min(lo, v), hi = max(hi, v);
            }
        }
        lo = __reduce_min_sync(RT_FULL, lo);
        hi = __reduce_max_sync(RT_FULL, hi);
        if ((threadIdx.x & 31) == 0) {
            red[0][threadIdx.x >> 5] = lo;
            red[1][threadIdx.x >> 5] = hi;
        }
        for (int k = threadIdx.x; k < kBinsLong; k += 256)
            hist[b * kBinsLong + k] = 0;
        const bool fits = tmp_off[b] + n <= scratch_cap;  // always, when the scratch holds all ids
        const int64_t nu = fits ? (n + kUnit - 1) / kUnit : 0;
        if (threadIdx.x == 0) {
            first = atomicAdd(hdr + HDR_UNITS, (unsigned long long)nu);
            if (!fits)
                atomicOr(flags, 1);
        }
        __syncthreads();
        for (int64_t u = threadIdx.x; u < nu; u += 256) {
            if ((int64_t)first + u < unit_cap)
                units[first + u] = Unit{(int32_t)b, (int32_t)u};
            else
                atomicOr(flags, 2);
        }
        if (threadIdx.x == 0) {
            for (int x = 0; x < 8; ++x)
                lo = min(lo, red[0][x]), hi = max(hi, red[1][x]);
            const BucketMap m = bucket_map(kBinsLong, lo, hi, nullptr);
            segs[b] = LongSeg{m.add, m.mult, 0};
        }
        __syncthreads();
    }
}

// The last range of rng[0 .. nr) that starts at or before place p (ranges
// ascend; the first starts at 0), found by the warp 32 probes at a time.
__device__ __forceinline__ int64_t range_at(const int2 *__restrict__ rng, int64_t nr, int p, int lane)
{
    int64_t lo = 0, hi = nr;  // the answer is in [lo, hi)
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t q = lo + lane * step;
        const unsigned m = __ballot_sync(RT_FULL, q < hi && rng[q].y <= p);
        const int64_t at = lo + (31 - __clz(m)) * step;  // lane 0's probe always holds
        hi = min(at + step, hi);
        lo = at;
    }
    return lo;
}

constexpr int kLongThreads = 256;

__global__ void __launch_bounds__(kLongThreads, 6)
    k_long_gather(const int32_t *__restrict__ list, const Unit *__restrict__ units,
                  const unsigned long long *__restrict__ n_units, int64_t unit_cap, const int64_t *__restrict__ off,
                  SortSources S, const LongSeg *__restrict__ segs, uint32_t *__restrict__ hist,
                  int32_t *__restrict__ out)
{
    __shared__ __align__(16) uint32_t buf[kUnit];
    __shared__ uint32_t bins[kBinsLong];
    constexpr int W = kLongThreads / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t cnt = list_len(n_units, unit_cap);
    for (int64_t u = blockIdx.x; u < cnt; u += gridDim.x) {
        const Unit un = units[u];
        const int32_t i = list[un.slot];
        const int64_t o = off[i], n = off[i + 1] - o;
        const int64_t p0 = (int64_t)un.part * kUnit, p1 = min(p0 + kUnit, n);
        const int64_t l0 = S.off_leaf[i], nl = leaf_end(S, i) - l0, nrl = n - nl;
        for (int k = threadIdx.x; k < kBinsLong; k += kLongThreads)
            bins[k] = 0;
        if (p1 > nrl) {  // leaf hits of the unit
            const int64_t a = max(p0, nrl);
            copy_async(buf + (a - p0), S.leaf + l0 + (a - nrl), (int)(p1 - a), threadIdx.x, kLongThreads);
        }
        if (p0 < nrl) {  // runs of the unit, a warp one after another
            const int64_t r0 = S.off_rng[i], nr = S.off_rng[i + 1] - r0;
            const int2 *rng = S.rng + r0;
            const int end = (int)min(p1, nrl);
            const int64_t first = range_at(rng, nr, (int)p0, lane), last = range_at(rng, nr, end - 1, lane);
            const int per = (int)((last - first + W) / W);  // runs of a warp
            const int64_t mine = min(first + (w + 1) * (int64_t)per, last + 1);
            for (int64_t rb = first + w * (int64_t)per; rb < mine; rb += 32) {
                const int2 g = rb + lane < nr ? rng[rb + lane] : make_int2(0, (int)nrl);
                const int after = rb + 32 < nr ? rng[rb + 32].y : (int)nrl;
                const int cnt = (int)min(mine - rb, (int64_t)32);
                for (int j = lane >> 4; j < cnt + (lane >> 4); j += 2) {  // 16 lanes a run
                    const int k = min(j, 31);
                    const int lo = __shfl_sync(RT_FULL, g.x, k), st = __shfl_sync(RT_FULL, g.y, k);
                    const int nx = __shfl_sync(RT_FULL, g.y, (k + 1) & 31);
                    const int a = max(st, (int)p0), e = min(k < 31 ? nx : after, end);
                    if (j < cnt && e > a)
                        copy_async(buf + (a - (int)p0), S.tree_ids + lo + (a - st), e - a, lane & 15, 16);
                }
            }
        }
        cp_async_wait();
        __syncthreads();
        const LongSeg sg = segs[un.slot];
        const int len = (int)(p1 - p0);
        for (int p = threadIdx.x; p < len; p += kLongThreads) {
            const int v = (int)buf[p];
            atomicAdd(&bins[bin_of(sg, v)], 1u);
            out[o + p0 + p] = v;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < kBinsLong; k += kLongThreads)
            if (bins[k])
                atomicAdd(hist + (int64_t)un.slot * kBinsLong + k, bins[k]);
        __syncthreads();
    }
}

// hist becomes the buckets' write cursors, table the bins' buckets.
__global__ void __launch_bounds__(kBinsLong)
    k_long_split(const int32_t *__restrict__ list, const unsigned long long *__restrict__ count, int64_t list_cap,
                 const int64_t *__restrict__ tmp_off, int64_t scratch_cap, const int64_t *__restrict__ off,
                 uint32_t *__restrict__ hist, uint16_t *__restrict__ table, SegDesc *__restrict__ buckets,
                 SegDesc *__restrict__ oversize, int64_t desc_cap, unsigned long long *__restrict__ hdr,
                 int32_t *__restrict__ flags)
{
    __shared__ uint32_t wsum[32], wfirst[32];
    __shared__ uint32_t starts[kBinsLong + 1];
    const int t = threadIdx.x;
    const int64_t cnt = list_len(count, list_cap);
    for (int64_t b = blockIdx.x; b < cnt; b += gridDim.x) {
        const int32_t seg = list[b];
        const int64_t o = off[seg], n = off[seg + 1] - o, tmp = tmp_off[b];
        if (tmp + n > scratch_cap)
            continue;
        const uint32_t c = hist[b * kBinsLong + t];
        int total;
        const uint32_t pre = (uint32_t)block_scan_int<kBinsLong>(wsum, (int)c, &total);
        // a bucket starts where another multiple of kBucketIds has been passed
        starts[t] = pre;
        __syncthreads();
        const bool head = t == 0 || pre / kBucketIds != starts[t - 1] / kBucketIds;
        int nb;
        const int k = block_scan_int<kBinsLong>(wfirst, head ? 1 : 0, &nb) + (head ? 0 : -1);  // this bin's bucket
        __syncthreads();
        if (head)
            starts[k] = pre;
        if (t == 0)
            starts[nb] = (uint32_t)n;
        table[b * kBinsLong + t] = (uint16_t)k;
        __syncthreads();
        if (t < nb) {
            const uint32_t s0 = starts[t], len = starts[t + 1] - s0;
            hist[b * kBinsLong + t] = s0;
            if (len > 0) {
                const SegDesc d{tmp + s0, o + s0, (int32_t)len, 0};
                const bool fits = len <= (uint32_t)kMidMax;
                const unsigned long long slot = atomicAdd(hdr + (fits ? HDR_BUCKETS : HDR_OVERSIZE), 1ull);
                if ((int64_t)slot < desc_cap)
                    (fits ? buckets : oversize)[slot] = d;
                else
                    atomicOr(flags, 2);
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kLongThreads, 6)
    k_long_scatter(const int32_t *__restrict__ list, const Unit *__restrict__ units,
                   const unsigned long long *__restrict__ n_units, int64_t unit_cap, const int64_t *__restrict__ off,
                   const int64_t *__restrict__ tmp_off, const LongSeg *__restrict__ segs,
                   uint32_t *__restrict__ cursors, const uint16_t *__restrict__ table,
                   const int32_t *__restrict__ ids, int32_t *__restrict__ scratch)
{
    __shared__ int32_t buf[kUnit];
    __shared__ uint16_t tab[kBinsLong];
    __shared__ uint32_t cnt_[kBinsLong];   // ids per bucket, then their cursors in buf
    __shared__ uint16_t from[kBinsLong];   // buckets' starts in buf
    __shared__ uint32_t to[kBinsLong];     // ... and in the segment's scratch
    __shared__ uint32_t wsum[32];
    constexpr int PER = kUnit / kLongThreads;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t total = list_len(n_units, unit_cap);
    for (int64_t u = blockIdx.x; u < total; u += gridDim.x) {
        const Unit un = units[u];
        const int32_t seg = list[un.slot];
        const int64_t o = off[seg], n = off[seg + 1] - o, tmp = tmp_off[un.slot];
        const int64_t p0 = (int64_t)un.part * kUnit;
        const int len = (int)min((int64_t)kUnit, n - p0);
        const LongSeg sg = segs[un.slot];
        const int nb = table[(int64_t)un.slot * kBinsLong + kBinsLong - 1] + 1;
        int v[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int p = k * kLongThreads + threadIdx.x;
            v[k] = p < len ? ids[o + p0 + p] : 0;
        }
        for (int k = threadIdx.x; k < kBinsLong; k += kLongThreads)
            tab[k] = table[(int64_t)un.slot * kBinsLong + k];
        for (int k = threadIdx.x; k < nb; k += kLongThreads)
            cnt_[k] = 0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (k * kLongThreads + (int)threadIdx.x < len)
                atomicAdd(&cnt_[tab[bin_of(sg, v[k])]], 1u);
        __syncthreads();
        // a few buckets a thread: places in buf, and a reservation in the scratch
        constexpr int MINE = kBinsLong / kLongThreads;
        const int k0 = MINE * threadIdx.x;
        uint32_t c[MINE], mine = 0;
#pragma unroll
        for (int k = 0; k < MINE; ++k) {
            c[k] = k0 + k < nb ? cnt_[k0 + k] : 0u;
            mine += c[k];
        }
        int sum;
        uint32_t at = (uint32_t)block_scan_int<kLongThreads>(wsum, (int)mine, &sum);
#pragma unroll
        for (int k = 0; k < MINE; ++k) {
            if (k0 + k < nb) {
                from[k0 + k] = (uint16_t)at;
                cnt_[k0 + k] = at;
                to[k0 + k] = c[k] ? atomicAdd(cursors + (int64_t)un.slot * kBinsLong + k0 + k, c[k]) : 0u;
                at += c[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (k * kLongThreads + (int)threadIdx.x < len)
                buf[atomicAdd(&cnt_[tab[bin_of(sg, v[k])]], 1u)] = v[k];
        __syncthreads();
        for (int k = w; k < nb; k += kLongThreads / 32) {  // cnt_[k] is now the run's end
            const uint32_t f = from[k], e = cnt_[k];
            int32_t *dst = scratch + tmp + to[k];
            for (uint32_t p = f + lane; p < e; p += 32)
                dst[p - f] = buf[p];
        }
        __syncthreads();
    }
}

// Fallback for buckets longer than kMidMax (heavily skewed ids): LSD radix
// sort through global memory from the bucket's scratch range to its
// place in the output, ping-ponging between the two.
__global__ void __launch_bounds__(256)
    k_sort_global(const SegDesc *__restrict__ list, const unsigned long long *__restrict__ count,
                  int64_t list_cap, int32_t *__restrict__ scratch, int32_t *__restrict__ ids)
{
    const int64_t cnt = list_len(count, list_cap);
    __shared__ uint32_t hist[kBins], run[kBins];
    __shared__ uint32_t red_and[8], red_or[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t b = blockIdx.x; b < cnt; b += gridDim.x) {
        const SegDesc d = list[b];
        uint32_t *x = reinterpret_cast<uint32_t *>(scratch) + d.src;
        uint32_t *y = reinterpret_cast<uint32_t *>(ids) + d.dst;  // output area
        const int64_t n = d.n;
        uint32_t a_and = 0xffffffffu, a_or = 0;
        for (int64_t p = threadIdx.x; p < n; p += 256) {
            a_and &= x[p];
            a_or |= x[p];
        }
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) {
            a_and &= __shfl_xor_sync(RT_FULL, a_and, q);
            a_or |= __shfl_xor_sync(RT_FULL, a_or, q);
        }
        if (lane == 0) {
            red_and[w] = a_and;
            red_or[w] = a_or;
        }
        __syncthreads();
        a_and = 0xffffffffu;
        a_or = 0;
        for (int q = 0; q < 8; ++q) {
            a_and &= red_and[q];
            a_or |= red_or[q];
        }
        const uint32_t diff = a_and ^ a_or;
        uint32_t *src = x, *dst = y;
        for (int shift = 0; shift < 32; shift += 8) {
            if (((diff >> shift) & 0xffu) == 0)
                continue;
            hist[threadIdx.x] = 0;
            __syncthreads();
            for (int64_t p = threadIdx.x; p < n; p += 256)
                atomicAdd(&hist[((src[p] ^ kSign) >> shift) & 0xffu], 1u);
            __syncthreads();
            if (threadIdx.x < 32) {
                uint32_t carry = 0;
                for (int c = 0; c < kBins; c += 32) {
                    const uint32_t v = hist[c + lane];
                    uint32_t inc = v;
#pragma unroll
                    for (int q = 1; q < 32; q <<= 1) {
                        const uint32_t u = __shfl_up_sync(RT_FULL, inc, q);
                        if (lane >= q)
                            inc += u;
                    }
                    run[c + lane] = carry + inc - v;
                    carry += __shfl_sync(RT_FULL, inc, 31);
                }
            }
            __syncthreads();
            // stable scatter: one warp walks the keys in order, 32 at a time
            if (w == 0) {
                const unsigned lt = lanemask_lt();
                for (int64_t p0 = 0; p0 < n; p0 += 32) {
                    const int64_t p = p0 + lane;
                    const bool ok = p < n;
                    const uint32_t k = ok ? src[p] : 0u;
                    const int dg = ok ? (int)(((k ^ kSign) >> shift) & 0xffu) : kBins;
                    const unsigned peers = __match_any_sync(RT_FULL, dg);
                    const uint32_t base = ok ? run[dg] : 0u;
                    if (ok)
                        dst[base + __popc(peers & lt)] = k;
                    __syncwarp();
                    if (ok && lane == __ffs(peers) - 1)
                        run[dg] = base + __popc(peers);
                    __syncwarp();
                }
            }
            __syncthreads();
            uint32_t *tmp = src;
            src = dst;
            dst = tmp;
        }
        if (src != y)
            for (int64_t p = threadIdx.x; p < n; p += 256)
                y[p] = src[p];
        __syncthreads();
    }
}

// --------------------------------------------------------------- launches
template <typename K>
rtree_status set_smem(K kern, size_t bytes)
{
    if (bytes > 48 * 1024)
        RT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return RTREE_OK;
}

struct Crowded {
    SegDesc *list;
    unsigned long long *count;
    int64_t cap;
};

template <int THREADS, int ITEMS, bool BUCKETS>
rtree_status launch_cta(const void *list, const unsigned long long *count, int64_t list_cap,
                        const int64_t *off, const SortSources &S, const int32_t *scratch,
                        int32_t *out, const Crowded &cr, unsigned long long *next, cudaStream_t s,
                        const char *name)
{
    if (list_cap <= 0)
        return RTREE_OK;
    auto kern = k_sort_cta<THREADS, ITEMS, BUCKETS>;
    const size_t bytes = sizeof(CtaSmem<THREADS, ITEMS>);
    RT_TRY(set_smem(kern, bytes));
    int per_sm = 0;
    RT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, THREADS, bytes));
    int64_t grid = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count();
    if (grid > list_cap)
        grid = list_cap;
    KernelTimer kt_(name, s);
    kern<<<(unsigned)grid, THREADS, bytes, s>>>(list, count, list_cap, off, S, scratch, out, cr.list,
                                                cr.count, cr.cap, next);
    RT_LAUNCH();
    return RTREE_OK;
}

template <int ITEMS>
rtree_status launch_lsd_of(const Crowded &cr, int least, int32_t *out, cudaStream_t s)
{
    const size_t bytes = sizeof(LsdSmem<ITEMS>);
    RT_TRY(set_smem(k_sort_lsd<ITEMS>, bytes));
    const int64_t grid = cr.cap < sm_count() ? cr.cap : sm_count();
    KernelTimer kt_("sort_lsd", s);
    k_sort_lsd<ITEMS><<<(unsigned)grid, 1024, bytes, s>>>(cr.list, cr.count, cr.cap, least, out);
    RT_LAUNCH();
    return RTREE_OK;
}

// The crowded segments of up to max_len ids.
rtree_status launch_lsd(const Crowded &cr, int64_t max_len, int32_t *out, cudaStream_t s)
{
    constexpr int small = 1024 * kLsdItems;
    static_assert(kCtaTop <= 2 * small, "the LSD fallback takes every CTA sort's segments");
    if (cr.cap <= 0)
        return RTREE_OK;
    RT_TRY(launch_lsd_of<kLsdItems>(cr, 0, out, s));
    return max_len > small ? launch_lsd_of<2 * kLsdItems>(cr, small + 1, out, s) : RTREE_OK;
}

rtree_status launch_warp(const int32_t *list, const unsigned long long *count, int64_t list_cap,
                         const int64_t *off, const SortSources &S, int32_t *out, cudaStream_t s)
{
    if (list_cap <= 0)
        return RTREE_OK;
    int64_t blocks = (list_cap + 7) / 8;
    const int64_t cap = (int64_t)sm_count() * 16;
    if (blocks > cap)
        blocks = cap;
    KernelTimer kt_("sort_warp", s);
    k_sort_warp<<<(unsigned)blocks, 256, 0, s>>>(list, count, list_cap, off, S, out);
    RT_LAUNCH();
    return RTREE_OK;
}

// Helper streams of this host thread on the current device, created on first
// use and kept for the thread's life: the sort's independent class kernels
// run on them beside the call's stream, so that one kernel's tail (its last
// CTAs finishing while the rest of the GPU idles) overlaps the next.
constexpr int kSide = 3;
struct SideStreams {
    int device = -1;
    cudaStream_t st[kSide] = {};
    cudaEvent_t ev[kSide + 1] = {};
};

rtree_status side_streams(SideStreams **out)
{
    constexpr int kMaxDev = 64;
    static thread_local SideStreams t_side[kMaxDev];
    int dev = 0;
    RT_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDev)
        return fail(RTREE_ECUDA, "device %d out of range", dev);
    SideStreams &sd = t_side[dev];
    if (sd.device != dev) {
        for (int i = 0; i < kSide; ++i)
            RT_CUDA(cudaStreamCreateWithFlags(&sd.st[i], cudaStreamNonBlocking));
        for (int i = 0; i <= kSide; ++i)
            RT_CUDA(cudaEventCreateWithFlags(&sd.ev[i], cudaEventDisableTiming));
        sd.device = dev;
    }
    *out = &sd;
    return RTREE_OK;
}

// Work enqueued on the side streams after begin() runs after everything
// enqueued on the main stream before it; the main stream waits for all of it
// when the Fork is joined or destroyed (also on an early error return, so
// that buffers freed in the main stream's order outlive their users).
// Declare it after every buffer the side work uses.
struct Fork {
    SideStreams *sd = nullptr;
    cudaStream_t s = nullptr;
    bool open = false;
    rtree_status begin(cudaStream_t main)
    {
        s = main;
        RT_TRY(side_streams(&sd));
        RT_CUDA(cudaEventRecord(sd->ev[kSide], s));
        for (int i = 0; i < kSide; ++i)
            RT_CUDA(cudaStreamWaitEvent(sd->st[i], sd->ev[kSide], 0));
        open = true;
        return RTREE_OK;
    }
    cudaStream_t side(int i) const { return sd->st[i]; }
    // The main stream waits for side stream i's work enqueued so far.
    rtree_status wait(int i)
    {
        RT_CUDA(cudaEventRecord(sd->ev[i], sd->st[i]));
        RT_CUDA(cudaStreamWaitEvent(s, sd->ev[i], 0));
        return RTREE_OK;
    }
    rtree_status join()
    {
        if (!open)
            return RTREE_OK;
        open = false;
        for (int i = 0; i < kSide; ++i)
            RT_TRY(wait(i));
        return RTREE_OK;
    }
    ~Fork()
    {
        if (open && join() != RTREE_OK)
            cudaGetLastError();
    }
};

}  // namespace

rtree_status segmented_sort_gather(int32_t *out, const int64_t *offsets, int64_t nseg, int64_t total,
                                   const SortSources &S, cudaStream_t s, int32_t *flags, int64_t out_cap,
                                   int64_t max_len, int64_t long_ids)
{
    if (nseg <= 0 || total <= 0)
        return RTREE_OK;
    if (max_len > total)
        max_len = total;
    if (out_cap < 0)
        out_cap = total;
    if (nseg >= (int64_t)INT32_MAX)
        return fail(RTREE_EOVERFLOW, "too many segments to sort (%lld)", (long long)nseg);
    // the whole sort, all classes, as one span (its kernels overlap)
    PhaseTimer span_("sort_all", s);
    // Every list length stays on the device; the launches below are sized
    // by upper bounds and read the actual lengths themselves, so the whole
    // sort is enqueued without a host round trip.
    const int64_t scratch_cap = long_ids < 0 || long_ids > total ? total : long_ids;
    const int64_t max_large = scratch_cap / (kCtaTop + 1) + 1 < nseg ? scratch_cap / (kCtaTop + 1) + 1 : nseg;
    // buckets: one per kBucketIds ids begun, and the last of each segment
    const int64_t desc_cap = 2 * max_large + scratch_cap / kBucketIds + 256;
    const int64_t unit_cap = max_large + scratch_cap / kUnit;
    DevBuf<int32_t> lists(s);
    DevBuf<int64_t> large_tmp(s);
    DevBuf<unsigned long long> hdr(s);
    RT_TRY(lists.alloc((size_t)C_COUNT * nseg, "sort lists"));
    RT_TRY(large_tmp.alloc(nseg, "sort lists"));
    // the header, two crowded-list counters, and one claim counter per CTA-sort launch
    constexpr int kClaims = 9;
    RT_TRY(hdr.alloc(HDR_WORDS + 2 + kClaims, "sort counters"));
    RT_CUDA(cudaMemsetAsync(hdr.p, 0, (HDR_WORDS + 2 + kClaims) * sizeof(unsigned long long), s));
    auto claim = [&](int k) { return hdr.p + HDR_WORDS + 2 + k; };
    const int sms = sm_count();
    {
        int64_t blocks = (nseg + 255) / 256;
        if (blocks > (int64_t)sms * 16)
            blocks = (int64_t)sms * 16;
        KernelTimer kt_("sort_classify", s);
        k_classify<<<(unsigned)blocks, 256, 0, s>>>(offsets, nseg, lists.p, nseg, large_tmp.p, hdr.p,
                                                    S, out, out_cap);
        RT_LAUNCH();
    }
    auto L = [&](int c) { return lists.p + (int64_t)c * nseg; };
    auto H = [&](int c) { return hdr.p + c; };
    // a class can hold at most total / (its smallest length) segments, and
    // none if no segment is that long
    auto cap_of = [&](int64_t min_len) {
        return min_len > max_len ? 0 : total / min_len < nseg ? total / min_len : nseg;
    };
    const int64_t cta_cap = cap_of(257);
    DevBuf<SegDesc> crowded(s);
    RT_TRY(crowded.alloc(cta_cap > 0 ? cta_cap : 1, "sort crowded list"));
    unsigned long long *n_crowded = hdr.p + HDR_WORDS;  // two counters after the header
    const Crowded cr1{crowded.p, n_crowded, cta_cap};
    const bool long_path = max_len > kCtaTop;  // else no segment can be long
    // the long path's buffers (segments over 32256 ids)
    DevBuf<int32_t> scratch(s);
    DevBuf<SegDesc> buckets(s), oversize(s), crowded2(s);
    DevBuf<LongSeg> long_segs(s);
    DevBuf<uint32_t> long_hist(s);
    DevBuf<uint16_t> long_table(s);
    DevBuf<Unit> units(s);
    if (long_path) {
        RT_TRY(scratch.alloc(scratch_cap, "sort scratch", long_ids >= 0 ? SCRATCH : EXACT));
        RT_TRY(buckets.alloc(desc_cap, "sort buckets"));
        RT_TRY(oversize.alloc(desc_cap, "sort buckets"));
        RT_TRY(crowded2.alloc(desc_cap, "sort crowded list"));
        RT_TRY(long_segs.alloc(max_large, "sort long segments"));
        RT_TRY(long_hist.alloc(max_large * kBinsLong, "sort long bins"));
        RT_TRY(long_table.alloc(max_large * kBinsLong, "sort long bins"));
        RT_TRY(units.alloc(unit_cap, "sort units"));
    }
    if (cta_cap == 0)  // short segments only: one kernel more
        return launch_warp(L(C_WARP), H(C_WARP), cap_of(2), offsets, S, out, s);
    // Three side streams and the call's stream run the classes side by side:
    //   side 2: the long path, a chain of small kernels, first to start;
    //   stream: the 32256-id CTA sort, the largest;
    //   side 1: the CTA sorts up to 16128 ids;
    //   side 0: those up to 2016 ids and the warp sort;
    // then, after all of them, the LSD fallback for crowded segments.  Larger
    // kernels are enqueued first so that smaller ones fill the SMs their last
    // CTAs leave idle.
    Fork fk;
    RT_TRY(fk.begin(s));
    const cudaStream_t s0 = fk.side(0), s1 = fk.side(1), s2 = fk.side(2);
    if (long_path) {
        const unsigned per_seg = (unsigned)(max_large < (int64_t)sms * 4 ? max_large : (int64_t)sms * 4);
        const unsigned per_unit = (unsigned)(unit_cap < (int64_t)sms * 6 ? unit_cap : (int64_t)sms * 6);
        {
            KernelTimer kt_("sort_long_plan", s2);
            k_long_plan<<<per_seg, 256, 0, s2>>>(L(C_LARGE), H(C_LARGE), max_large, large_tmp.p, scratch_cap, offsets, S,
                                                 long_segs.p, long_hist.p, units.p, unit_cap, hdr.p, flags);
            RT_LAUNCH();
        }
        {
            KernelTimer kt_("sort_long_gather", s2);
            k_long_gather<<<per_unit, kLongThreads, 0, s2>>>(L(C_LARGE), units.p, H(HDR_UNITS), unit_cap, offsets, S,
                                                             long_segs.p, long_hist.p, out);
            RT_LAUNCH();
        }
        {
            KernelTimer kt_("sort_long_split", s2);
            k_long_split<<<per_seg, kBinsLong, 0, s2>>>(L(C_LARGE), H(C_LARGE), max_large, large_tmp.p, scratch_cap,
                                                        offsets, long_hist.p, long_table.p, buckets.p, oversize.p,
                                                        desc_cap, hdr.p, flags);
            RT_LAUNCH();
        }
        {
            KernelTimer kt_("sort_long_scatter", s2);
            k_long_scatter<<<per_unit, kLongThreads, 0, s2>>>(L(C_LARGE), units.p, H(HDR_UNITS), unit_cap, offsets,
                                                              large_tmp.p, long_segs.p, long_hist.p, long_table.p, out,
                                                              scratch.p);
            RT_LAUNCH();
        }
        const Crowded cr2{crowded2.p, n_crowded + 1, desc_cap};
        RT_TRY((launch_cta<512, 32, true>(buckets.p, H(HDR_BUCKETS), desc_cap, nullptr, S, scratch.p, out, cr2, claim(1), s2, "sort_bucket")));
        RT_TRY(launch_lsd(cr2, kMidMax, out, s2));
        {
            int64_t g2 = desc_cap < (int64_t)sms * 4 ? desc_cap : (int64_t)sms * 4;
            KernelTimer kt_("sort_global", s2);
            k_sort_global<<<(unsigned)g2, 256, 0, s2>>>(oversize.p, H(HDR_OVERSIZE), desc_cap, scratch.p,
                                                        out);
            RT_LAUNCH();
        }
    }
    RT_TRY((launch_cta<1024, 32, false>(L(C_CTA32K), H(C_CTA32K), cap_of(kMidMax + 1), offsets, S, nullptr, out, cr1, claim(0), s, "sort_cta")));
    RT_TRY((launch_cta<512, 32, false>(L(C_CTA16K), H(C_CTA16K), cap_of(cta_ids(512, 16) + 1), offsets, S, nullptr, out, cr1, claim(2), s1, "sort_cta")));
    RT_TRY((launch_cta<512, 16, false>(L(C_CTA8K), H(C_CTA8K), cap_of(cta_ids(256, 16) + 1), offsets, S, nullptr, out, cr1, claim(3), s1, "sort_cta")));
    RT_TRY((launch_cta<256, 16, false>(L(C_CTA4K), H(C_CTA4K), cap_of(cta_ids(128, 16) + 1), offsets, S, nullptr, out, cr1, claim(4), s1, "sort_cta")));
    RT_TRY((launch_cta<128, 16, false>(L(C_CTA2K), H(C_CTA2K), cap_of(cta_ids(64, 16) + 1), offsets, S, nullptr, out, cr1, claim(5), s0, "sort_cta")));
    RT_TRY((launch_cta<64, 16, false>(L(C_CTA1K), H(C_CTA1K), cap_of(257), offsets, S, nullptr, out, cr1, claim(8), s0, "sort_cta")));
    RT_TRY(launch_warp(L(C_WARP), H(C_WARP), cap_of(2), offsets, S, out, s0));
    RT_TRY(fk.join());
    return launch_lsd(cr1, max_len, out, s);
}

}  // namespace rt
