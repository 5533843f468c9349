// radix_sort.cu -- stable LSD radix sort of (uint32 key, uint32 value) pairs.
//
// Used by the STR bulk load (sort by centre key, then by slab), by the query
// ordering and by the join (lexicographic sort of result pairs).  Small sorts
// are one launch of a cluster (below); otherwise each 8-bit digit pass is reduce-then-scan over a persistent grid of G CTAs, each
// owning a contiguous run of 4096-item tiles:
//   k_hist     CTA c counts the digits of its run: hist[d * G + c];
//   k_scan     one CTA per digit scans its row: offs[d * G + c] = items of
//              digit d in CTAs before c, and the digit's total;
//   k_scatter  CTA c walks its tiles in order, keeping a running offset per
//              digit: each tile is ranked in shared memory and written out
//              one digit run after another.
// No CTA waits for another.  Stability: items are ranked in input order
// inside a tile (each warp owns a contiguous run of the tile and walks it 32
// items at a time; lanes holding the same digit find each other with one
// ballot per digit bit and rank by lane order on top of a per-warp running
// count), tiles are taken in order inside a CTA, and CTAs own consecutive
// runs.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "internal.cuh"

namespace rt {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 16;
constexpr int kTile = kThreads * kItems;  // 4096
constexpr int kBins = 256;
constexpr int kWide = 1024;               // digits of up to 10 bits, where they save a pass
constexpr int kWarpRun = 32 * kItems;     // contiguous items owned by one warp
static_assert(kThreads == kBins, "one thread per digit");

// A number of each device, worked out at its first use there: how many CTAs of a
// kernel fit, after the kernel's attributes have been set (which CUDA keeps per
// device too, so a number of the whole process would leave the others without).
class PerDevice {
    static constexpr int kMaxDev = 64;
    std::once_flag once_[kMaxDev];
    int value_[kMaxDev] = {};

public:
    template <typename F>
    int get(F f)
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
            cudaGetLastError();
            return f();
        }
        std::call_once(once_[dev], [&] { value_[dev] = f(); });
        return value_[dev];
    }
};

// Tiles [t0, t1) of CTA c out of G (balanced: they differ by at most one).
__device__ __forceinline__ void run_of(int64_t ntiles, int G, int c, int64_t &t0, int64_t &t1)
{
    t0 = ntiles * c / G;
    t1 = ntiles * (c + 1) / G;
}

// Lanes of the warp whose digit equals this lane's (all lanes valid or not
// take part; the answer is meaningful for valid lanes), from one ballot per
// digit bit.
template <int BITS = 8>
__device__ __forceinline__ unsigned peers_of(int dg, uint32_t mask, bool ok)
{
    unsigned peers = __ballot_sync(RT_FULL, ok);
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
        if (!((mask >> b) & 1u))
            break;
        const unsigned m = __ballot_sync(RT_FULL, (dg >> b) & 1);
        peers &= (dg >> b) & 1 ? m : ~m;
    }
    return peers;
}

// Exclusive scan of one value per thread across the block (wsum: one word
// per warp of shared memory); every thread gets its prefix.
template <int THREADS>
__device__ __forceinline__ uint32_t block_excl(uint32_t v, uint32_t *wsum)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(RT_FULL, inc, o);
        if (lane >= o)
            inc += u;
    }
    if (lane == 31)
        wsum[w] = inc;
    __syncthreads();
    uint32_t add = 0;
    for (int x = 0; x < w; ++x)
        add += wsum[x];
    __syncthreads();
    return add + inc - v;
}

template <int BINS>
__global__ void __launch_bounds__(kThreads) k_hist(const uint32_t *__restrict__ keys, int64_t n,
                                                   int shift, uint32_t mask, int64_t ntiles, int G,
                                                   uint32_t *__restrict__ hist)
{
    __shared__ uint32_t h[kWarps][BINS];
    for (int i = threadIdx.x; i < kWarps * BINS; i += kThreads)
        (&h[0][0])[i] = 0;
    __syncthreads();
    int64_t t0, t1;
    run_of(ntiles, G, blockIdx.x, t0, t1);
    const int64_t b = t0 * kTile, e = t1 * kTile < n ? t1 * kTile : n;
    const int w = threadIdx.x >> 5;
#pragma unroll 8
    for (int64_t k = b + threadIdx.x; k < e; k += kThreads)
        atomicAdd(&h[w][(__ldg(keys + k) >> shift) & mask], 1u);
    __syncthreads();
#pragma unroll
    for (int d = threadIdx.x; d < BINS; d += kThreads) {
        uint32_t s = 0;
#pragma unroll
        for (int x = 0; x < kWarps; ++x)
            s += h[x][d];
        hist[(int64_t)d * G + blockIdx.x] = s;
    }
}

// Per digit d (one CTA each): exclusive scan of hist[d*G .. d*G+G) into
// offs (the digit's CTAs in order) and the digit's total into tot[d].
__global__ void __launch_bounds__(kThreads) k_scan(const uint32_t *__restrict__ hist, int G,
                                                   uint32_t *__restrict__ offs, uint32_t *__restrict__ tot)
{
    __shared__ uint32_t wsum[kWarps];
    const int64_t row = (int64_t)blockIdx.x * G;
    const int per = (G + kThreads - 1) / kThreads;
    const int lo = threadIdx.x * per, hi = lo + per < G ? lo + per : G;
    uint32_t s = 0;
    for (int i = lo; i < hi; ++i)
        s += hist[row + i];
    const uint32_t before = block_excl<kThreads>(s, wsum);
    uint32_t run = before;
    for (int i = lo; i < hi; ++i) {
        const uint32_t v = hist[row + i];
        offs[row + i] = run;
        run += v;
    }
    if (threadIdx.x == kThreads - 1)
        tot[blockIdx.x] = run;
}

// What the last pass leaves.
enum : int {
    END_PAIRS = 0,    // the sorted keys and values
    END_VALUES = 1,   // the values
    END_GROUPS = 2,   // table[value] = place / size, nothing else
    END_RELABEL = 3   // the values, and table[value] as their keys
};
struct RadixEnd {
    int what;
    uint32_t *table;
    uint32_t size;
};

template <int BINS>
struct ScatterSmem {
    // counts of a tile and places in it fit 16 bits; the narrow form has room for words
    using Count = typename std::conditional<(BINS > kBins), uint16_t, uint32_t>::type;
    uint32_t k[kTile], v[kTile];
    uint32_t base[BINS];  // where this CTA's next item of each digit goes
    uint32_t wsum[kWarps];
    Count wcnt[kWarps][BINS];
    Count tstart[BINS];
};

// Four CTAs per SM (64 registers a thread): the tiles' loads of one CTA
// overlap the ranking of the others.  A value is its own index where vin is null.
template <int BINS, int END>
__global__ void __launch_bounds__(kThreads, 4)
    k_scatter(const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin,
              uint32_t *__restrict__ kout, uint32_t *__restrict__ vout, int64_t n, int shift,
              uint32_t mask, const uint32_t *__restrict__ offs, const uint32_t *__restrict__ tot,
              int64_t ntiles, int G, RadixEnd end)
{
    constexpr int PER = BINS / kThreads;  // digits a thread looks after
    using Smem = ScatterSmem<BINS>;
    using Count = typename Smem::Count;
    extern __shared__ uint4 smem[];
    Smem &sm = *reinterpret_cast<Smem *>(smem);

    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, d0 = threadIdx.x * PER;
    const unsigned lt = lanemask_lt();
    int64_t t0, t1;
    run_of(ntiles, G, blockIdx.x, t0, t1);
    // items of smaller digits come first, then this digit's items of earlier CTAs
    {
        uint32_t all = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j)
            all += tot[d0 + j];
        uint32_t at = block_excl<kThreads>(all, sm.wsum);
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            sm.base[d0 + j] = at + offs[(int64_t)(d0 + j) * G + blockIdx.x];
            at += tot[d0 + j];
        }
    }
    for (int64_t tile = t0; tile < t1; ++tile) {
        for (int i = threadIdx.x; i < (int)(sizeof(sm.wcnt) / 4); i += kThreads)
            reinterpret_cast<uint32_t *>(&sm.wcnt[0][0])[i] = 0;
        __syncthreads();  // also: the previous tile's staging is written out

        const int64_t tile0 = tile * kTile;
        const int64_t wbase = tile0 + (int64_t)w * kWarpRun;
        uint32_t k[kItems], rank[kItems];
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const int64_t idx = wbase + i * 32 + lane;
            k[i] = idx < n ? __ldg(kin + idx) : 0u;
        }
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const bool ok = wbase + i * 32 + lane < n;
            const int dg = (int)((k[i] >> shift) & mask);
            const unsigned peers = peers_of<(BINS > kBins ? 10 : 8)>(dg, mask, ok);
            const uint32_t prev = ok ? sm.wcnt[w][dg] : 0u;
            rank[i] = prev + __popc(peers & lt);
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1)
                sm.wcnt[w][dg] = (Count)(prev + __popc(peers));
            __syncwarp();
        }
        __syncthreads();

        // per digit: exclusive prefix over warps (in place) and the tile's count
        uint32_t cnt[PER], all = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            cnt[j] = 0;
#pragma unroll
            for (int x = 0; x < kWarps; ++x) {
                const uint32_t c = sm.wcnt[x][d0 + j];
                sm.wcnt[x][d0 + j] = (Count)cnt[j];
                cnt[j] += c;
            }
            all += cnt[j];
        }
        uint32_t at = block_excl<kThreads>(all, sm.wsum);  // the digit runs' starts in the tile
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            sm.tstart[d0 + j] = (Count)at;
            at += cnt[j];
        }
        __syncthreads();

        // stage the tile in digit order: keys, then values (read only now)
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            if (wbase + i * 32 + lane < n) {
                const int dg = (int)((k[i] >> shift) & mask);
                rank[i] += sm.tstart[dg] + sm.wcnt[w][dg];
                sm.k[rank[i]] = k[i];
            }
        }
        if (vin) {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const int64_t idx = wbase + i * 32 + lane;
                if (idx < n)
                    sm.v[rank[i]] = __ldg(vin + idx);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const int64_t idx = wbase + i * 32 + lane;
                if (idx < n)
                    sm.v[rank[i]] = (uint32_t)idx;
            }
        }
        __syncthreads();
        const int tn = (int)(n - tile0 < kTile ? n - tile0 : kTile);
        for (int p = threadIdx.x; p < tn; p += kThreads) {
            const uint32_t key = sm.k[p];
            const int dd = (int)((key >> shift) & mask);
            const uint32_t dst = sm.base[dd] + (uint32_t)p - sm.tstart[dd];
            if (dst < (uint64_t)n) {
                if (END == END_PAIRS)
                    kout[dst] = key;
                const uint32_t value = sm.v[p];
                if (END == END_GROUPS) {
                    if (value < (uint64_t)n)
                        end.table[value] = dst / end.size;
                } else {
                    vout[dst] = value;
                }
                if (END == END_RELABEL)
                    kout[dst] = value < (uint64_t)n ? __ldg(end.table + value) : 0u;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PER; ++j)
            sm.base[d0 + j] += cnt[j];
    }
}

// CTAs of the persistent grid: every SM full (at most one tile each).
template <int BINS, int END>
int grid_for(int64_t ntiles)
{
    static PerDevice ctas;
    const int per_sm = ctas.get([] {
        int v = 0;
        if (cudaFuncSetAttribute(k_scatter<BINS, END>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(ScatterSmem<BINS>)) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_scatter<BINS, END>, kThreads,
                                                          sizeof(ScatterSmem<BINS>)) != cudaSuccess || v < 1) {
            cudaGetLastError();
            v = 1;
        }
        return v;
    });
    const int64_t g = (int64_t)per_sm * sm_count();
    return (int)(ntiles < g ? ntiles : g);
}

// Words of digit counts that a pass over n pairs needs.
template <int BINS, int END>
size_t count_words(int64_t n)
{
    return (size_t)BINS * (2 * grid_for<BINS, END>((n + kTile - 1) / kTile) + 1);
}

// One pass: digit (key >> shift) & mask, of at most BINS values.
template <int BINS, int END>
rtree_status radix_pass(const uint32_t *kin, const uint32_t *vin, uint32_t *kout, uint32_t *vout, int64_t n,
                        int shift, uint32_t mask, const RadixEnd &end, uint32_t *counts, cudaStream_t s)
{
    const int64_t ntiles = (n + kTile - 1) / kTile;
    const int G = grid_for<BINS, END>(ntiles);
    uint32_t *hist = counts, *offs = hist + (size_t)BINS * G, *tot = offs + (size_t)BINS * G;
    {
        KernelTimer kt_("hist", s);
        k_hist<BINS><<<(unsigned)G, kThreads, 0, s>>>(kin, n, shift, mask, ntiles, G, hist);
        RT_LAUNCH();
    }
    {
        KernelTimer kt_("radix_scan", s);
        k_scan<<<BINS, kThreads, 0, s>>>(hist, G, offs, tot);
        RT_LAUNCH();
    }
    KernelTimer kt_("scatter", s);
    k_scatter<BINS, END><<<(unsigned)G, kThreads, sizeof(ScatterSmem<BINS>), s>>>(
        kin, vin, kout, vout, n, shift, mask, offs, tot, ntiles, G, end);
    RT_LAUNCH();
    return RTREE_OK;
}

// All passes over the bits [bit_lo, bit_hi); the last one leaves END.
template <int END>
rtree_status radix_passes(const uint32_t *kin, const uint32_t *vin, uint32_t *kout, uint32_t *vout, int64_t n,
                          int bit_lo, int bit_hi, const RadixEnd &end, cudaStream_t s)
{
    // ten bits at a time where that saves a pass (10M items by 9 bits: 90 us less than two
    // passes take)
    const int bits = bit_hi - bit_lo, wide = (bits + 9) / 10, passes = (bits + 7) / 8 > wide ? wide : (bits + 7) / 8;
    const int digit = (bits + passes - 1) / passes;
    DevBuf<uint32_t> tk(s), tv(s), counts(s);
    if (passes > 1) {
        RT_TRY(tk.alloc(n, "radix keys"));
        RT_TRY(tv.alloc(n, "radix values"));
    }
    const size_t words = digit > 8 ? std::max(count_words<kWide, END>(n), count_words<kWide, END_PAIRS>(n))
                                   : std::max(count_words<kBins, END>(n), count_words<kBins, END_PAIRS>(n));
    RT_TRY(counts.alloc(words, "radix digit counts"));
    // Ping-pong so that the last pass writes kout/vout.
    uint32_t *bk[2] = {kout, tk.p}, *bv[2] = {vout, tv.p};
    for (int p = 0; p < passes; ++p) {
        const int shift = bit_lo + digit * p, o = (passes - 1 - p) & 1;
        const uint32_t mask = (1u << min(digit, bit_hi - shift)) - 1u;
        const bool last = p == passes - 1;
        rtree_status st;
        if (digit > 8)
            st = last ? radix_pass<kWide, END>(kin, vin, bk[o], bv[o], n, shift, mask, end, counts.p, s)
                      : radix_pass<kWide, END_PAIRS>(kin, vin, bk[o], bv[o], n, shift, mask, end, counts.p, s);
        else
            st = last ? radix_pass<kBins, END>(kin, vin, bk[o], bv[o], n, shift, mask, end, counts.p, s)
                      : radix_pass<kBins, END_PAIRS>(kin, vin, bk[o], bv[o], n, shift, mask, end, counts.p, s);
        RT_TRY(st);
        kin = bk[o];
        vin = bv[o];
    }
    return RTREE_OK;
}

// ---- small sorts: every pass in one launch, by a cluster of CTAs.
// A pass over up to a few hundred thousand pairs takes a few microseconds; as
// three launches it takes about 20.  The CTAs own consecutive chunks and meet
// twice a pass at the cluster's barrier: once to read each other's digit counts
// (from shared memory), once so that the next pass reads what this one wrote.
// Sorting 2,000 pairs by 32 bits takes 28 us instead of 97, 100K 51 instead of
// 104, 200K 71 instead of 105 (a pass's kernels summed), and the sort of 400K
// would take 125 instead of 105: its 16 SMs are then short of issue slots.
// The first pass can make its keys itself, and the last one can keep less than
// the sorted pairs, so that a level of a tree is packed by two launches.
constexpr int kCThreads = 1024;
constexpr int kCWarps = kCThreads / 32;
constexpr int kCItems = 16;
constexpr int kCTile = kCThreads * kCItems;
constexpr int kCluster = 16;
constexpr int64_t kClusterMost = (int64_t)1 << 18;

enum : int {
    SRC_PAIRS = 0,  // keys kin, values vin
    SRC_BOXES = 1,  // the centre keys of boxes along `axis`, values their indices
    SRC_TABLE = 2   // values vin, keys table[value]
};

struct ClusterSort {
    const uint32_t *kin, *vin;
    const float4 *boxes;
    const uint32_t *table;
    uint32_t *k[2], *v[2];  // the passes' outputs in turn, the last one's first
    uint32_t *group;        // if given, the last pass writes group[value] = place / size only
    uint32_t size;
    int axis, n, bit_lo, bit_hi, passes;
    int keys_out;  // the last pass writes the keys too
};

struct ClusterSmem {
    uint32_t k[kCTile], v[kCTile];
    uint32_t wcnt[kCWarps][kBins];
    uint32_t part[kCThreads];
    uint32_t hist[kBins];  // this CTA's items of each digit (the cluster reads it)
    uint32_t base[kBins], tstart[kBins];
    uint32_t wsum[2][kWarps];
};

__device__ __forceinline__ void cluster_arrive()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The word of CTA `rank`'s shared memory at the place that p has in this one's.
__device__ __forceinline__ uint32_t cluster_load(const uint32_t *p, unsigned rank)
{
    uint32_t at = (uint32_t)__cvta_generic_to_shared(p), v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(at), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}

// Exclusive scan over the first kBins threads; the others get no answer.
__device__ __forceinline__ uint32_t bins_excl(uint32_t v, uint32_t *wsum)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(RT_FULL, inc, o);
        if (lane >= o)
            inc += u;
    }
    if (lane == 31 && w < kWarps)
        wsum[w] = inc;
    __syncthreads();
    uint32_t add = 0;
#pragma unroll
    for (int x = 0; x < kWarps; ++x)
        add += x < w ? wsum[x] : 0u;
    return add + inc - v;
}

// Sort blockIdx.x / (CTAs of a cluster) of the launch: a, or b.
template <int SRC>
__global__ void __launch_bounds__(kCThreads, 1)
    k_sort_cluster(const __grid_constant__ ClusterSort first, const __grid_constant__ ClusterSort second)
{
    extern __shared__ uint4 smem[];
    ClusterSmem &sm = *reinterpret_cast<ClusterSmem *>(smem);
    unsigned me, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(me));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const ClusterSort &a = blockIdx.x < C ? first : second;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31, d = t & (kBins - 1), quarter = t / kBins;
    const unsigned lt = lanemask_lt();
    // chunks, and the tiles of one, are equal but for the last
    const int n = a.n, chunk = (int)((((int64_t)n + C - 1) / C + 31) / 32 * 32);
    const int64_t begin = (int64_t)me * chunk;
    const int b = (int)(begin < n ? begin : n);
    const int len = min(chunk, n - b), e = b + len;
    const int tiles = max(1, (len + kCTile - 1) / kCTile);
    const int per = (len + tiles * kCThreads - 1) / (tiles * kCThreads);  // items a thread has of a tile

    const uint32_t *kin = a.kin, *vin = a.vin;
    for (int p = 0; p < a.passes; ++p) {
        const int shift = a.bit_lo + 8 * p;
        const uint32_t mask = (1u << min(8, a.bit_hi - shift)) - 1u;
        uint32_t *kout = a.k[(a.passes - 1 - p) & 1], *vout = a.v[(a.passes - 1 - p) & 1];
        const bool last = p == a.passes - 1;
        auto key_of = [&](int i) -> uint32_t {
            if (SRC == SRC_BOXES && p == 0) {
                const float4 box = __ldg(a.boxes + i);
                return a.axis == 0 ? centre_key(box.x, box.z) : centre_key(box.y, box.w);
            }
            if (SRC == SRC_TABLE && p == 0) {
                const uint32_t v = __ldcg(vin + i);
                return v < (uint32_t)n ? __ldcg(a.table + v) : 0u;
            }
            return __ldcg(kin + i);
        };
        if (tiles > 1) {  // the digits of all tiles are counted first
            for (int i = t; i < kCWarps * kBins; i += kCThreads)
                (&sm.wcnt[0][0])[i] = 0;
            __syncthreads();
#pragma unroll 8
            for (int i = b + t; i < e; i += kCThreads)
                atomicAdd(&sm.wcnt[w][(key_of(i) >> shift) & mask], 1u);
            __syncthreads();
            uint32_t s = 0;
#pragma unroll
            for (int x = 0; x < kCWarps; x += 4)
                s += sm.wcnt[x + quarter][d];
            sm.part[t] = s;
            __syncthreads();
            if (t < kBins)
                sm.hist[t] = sm.part[t] + sm.part[t + kBins] + sm.part[t + 2 * kBins] + sm.part[t + 3 * kBins];
        }
        for (int tile = 0; tile < tiles; ++tile) {
            const int tile0 = b + tile * per * kCThreads;
            const int wbase = tile0 + w * per * 32;
            uint32_t k[kCItems], rank[kCItems];
#pragma unroll
            for (int i = 0; i < kCItems; ++i) {
                const int idx = wbase + i * 32 + lane;
                k[i] = i < per && idx < e ? key_of(idx) : 0u;
            }
            for (int i = lane; i < kBins; i += 32)  // the warp's own counts
                sm.wcnt[w][i] = 0;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kCItems; ++i) {
                if (i >= per)
                    break;
                const bool ok = wbase + i * 32 + lane < e;
                const int dg = (int)((k[i] >> shift) & mask);
                const unsigned peers = peers_of(dg, mask, ok);
                const uint32_t prev = ok ? sm.wcnt[w][dg] : 0u;
                rank[i] = prev + __popc(peers & lt);
                __syncwarp();
                if (ok && lane == __ffs(peers) - 1)
                    sm.wcnt[w][dg] = prev + __popc(peers);
                __syncwarp();
            }
            __syncthreads();  // also: the tile before is written out, its base advanced
            // per digit: exclusive prefix over warps (in place) and the tile's count
            constexpr int kQ = kCWarps / 4;  // warps per quarter
            uint32_t c[kQ], s = 0;
#pragma unroll
            for (int x = 0; x < kQ; ++x) {
                c[x] = sm.wcnt[quarter * kQ + x][d];
                s += c[x];
            }
            sm.part[t] = s;
            __syncthreads();
            uint32_t run = 0, cnt = 0;
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t v = sm.part[x * kBins + d];
                run += x < quarter ? v : 0u;
                cnt += v;
            }
            if (tile == 0) {
                if (tiles == 1 && t < kBins)
                    sm.hist[t] = cnt;
                cluster_arrive();
            }
#pragma unroll
            for (int x = 0; x < kQ; ++x) {
                sm.wcnt[quarter * kQ + x][d] = run;
                run += c[x];
            }
            const uint32_t at = bins_excl(cnt, sm.wsum[0]);
            if (t < kBins)
                sm.tstart[t] = at;
            if (tile == 0) {
                cluster_wait();
                uint32_t mine = 0, all = 0;
                if (t < kBins) {
#pragma unroll
                    for (unsigned r = 0; r < kCluster; ++r) {
                        const uint32_t v = r < C ? cluster_load(&sm.hist[t], r) : 0u;
                        mine += r < me ? v : 0u;
                        all += v;
                    }
                }
                const uint32_t smaller = bins_excl(all, sm.wsum[1]);
                if (t < kBins)
                    sm.base[t] = smaller + mine;
            }
            __syncthreads();
            // stage the tile in digit order: keys, then values
#pragma unroll
            for (int i = 0; i < kCItems; ++i) {
                if (i < per && wbase + i * 32 + lane < e) {
                    const int dg = (int)((k[i] >> shift) & mask);
                    rank[i] += sm.tstart[dg] + sm.wcnt[w][dg];
                    sm.k[rank[i]] = k[i];
                }
            }
#pragma unroll
            for (int i = 0; i < kCItems; ++i) {
                const int idx = wbase + i * 32 + lane;
                if (i < per && idx < e)
                    sm.v[rank[i]] = SRC == SRC_BOXES && p == 0 ? (uint32_t)idx : __ldcg(vin + idx);
            }
            __syncthreads();
            const int tn = min(per * kCThreads, e - tile0);
            for (int i = t; i < tn; i += kCThreads) {
                const uint32_t key = sm.k[i], value = sm.v[i];
                const int dg = (int)((key >> shift) & mask);
                const uint32_t dst = sm.base[dg] + (uint32_t)i - sm.tstart[dg];
                if (dst >= (uint32_t)n)
                    continue;
                if (last && a.group) {
                    if (value < (uint32_t)n)
                        a.group[value] = dst / a.size;
                    continue;
                }
                vout[dst] = value;
                if (!last || a.keys_out)
                    kout[dst] = key;
            }
            if (tile + 1 < tiles) {
                __syncthreads();
                if (t < kBins)
                    sm.base[t] += cnt;
            }
        }
        cluster_arrive();  // the outputs are written; the digit counts are read
        cluster_wait();
        kin = kout;
        vin = vout;
    }
}

// A launch of k_sort_cluster; at is what it refers to.
void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at, int C, int clusters, cudaStream_t s)
{
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(C * clusters);
    cfg.blockDim = dim3(kCThreads);
    cfg.dynamicSmemBytes = sizeof(ClusterSmem);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
}

template <int SRC>
bool cluster_fits(int C)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at{};
    cluster_config(cfg, at, C, 1, nullptr);
    int fit = 0;
    if (cudaFuncSetAttribute(k_sort_cluster<SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(ClusterSmem)) == cudaSuccess &&
        cudaFuncSetAttribute(k_sort_cluster<SRC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&fit, k_sort_cluster<SRC>, &cfg) == cudaSuccess && fit > 0)
        return true;
    cudaGetLastError();
    return false;
}

// CTAs a cluster can have on the current device (16, 8, or 0 if there is none).
int cluster_ctas()
{
    static PerDevice most;
    return most.get([] {
        for (int c = kCluster; c >= 8; c >>= 1)
            if (cluster_fits<SRC_PAIRS>(c) && cluster_fits<SRC_BOXES>(c) && cluster_fits<SRC_TABLE>(c))
                return c;
        return 0;
    });
}

template <int SRC>
rtree_status launch_cluster(const ClusterSort &a, const ClusterSort &b, int clusters, cudaStream_t s)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at{};
    cluster_config(cfg, at, cluster_ctas(), clusters, s);
    KernelTimer kt_("sort_cluster", s);
    RT_CUDA(cudaLaunchKernelEx(&cfg, k_sort_cluster<SRC>, a, b));
    RT_LAUNCH();
    return RTREE_OK;
}

}  // namespace

rtree_status radix_sort_pairs(const uint32_t *kin, const uint32_t *vin, uint32_t *kout,
                              uint32_t *vout, int64_t n, int bit_lo, int bit_hi, cudaStream_t s)
{
    if (n <= 0)
        return RTREE_OK;
    if (n >= (int64_t)1 << 31)
        return fail(RTREE_EOVERFLOW, "radix sort of %lld items exceeds 2^31", (long long)n);
    if (bit_hi <= bit_lo) {
        RT_CUDA(cudaMemcpyAsync(kout, kin, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
        RT_CUDA(cudaMemcpyAsync(vout, vin, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
        return RTREE_OK;
    }
    if (n <= kClusterMost && cluster_ctas() > 0) {
        const int passes = (bit_hi - bit_lo + 7) / 8;
        DevBuf<uint32_t> tk(s), tv(s);
        if (passes > 1) {
            RT_TRY(tk.alloc(n, "radix keys"));
            RT_TRY(tv.alloc(n, "radix values"));
        }
        const ClusterSort a{kin, vin, nullptr, nullptr, {kout, tk.p}, {vout, tv.p}, nullptr, 1,
                            0, (int)n, bit_lo, bit_hi, passes, 1};
        return launch_cluster<SRC_PAIRS>(a, a, 1, s);
    }
    return radix_passes<END_PAIRS>(kin, vin, kout, vout, n, bit_lo, bit_hi, RadixEnd{END_PAIRS, nullptr, 1}, s);
}

namespace {

// Both centre keys of every box, read once.
__global__ void k_keys(const float4 *__restrict__ boxes, int64_t m, uint32_t *__restrict__ kx,
                       uint32_t *__restrict__ ky)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float4 b = boxes[i];
        kx[i] = centre_key(b.x, b.z);
        ky[i] = centre_key(b.y, b.w);
    }
}

// Slabs by the whole chip's passes: the x sort's last pass writes the items'
// slabs, the y sort's last pass looks them up as the keys of the third sort.
// Apart, the passes that made the keys of each axis, the slabs and the third
// sort's keys cost a 10M-box build 200 us of 2,290.
rtree_status str_order_large(const float4 *boxes, int64_t m, uint32_t size, int bits, uint32_t *pack, cudaStream_t s)
{
    DevBuf<uint32_t> kx(s), ky(s), k(s), v(s);
    RT_TRY(kx.alloc(m, "build keys"));
    RT_TRY(ky.alloc(m, "build keys"));
    RT_TRY(k.alloc(m, "build keys"));
    RT_TRY(v.alloc(m, "build values"));
    {
        KernelTimer kt_("keys", s);
        const int64_t blocks = (m + kThreads - 1) / kThreads;
        k_keys<<<(unsigned)(blocks < 1048576 ? blocks : 1048576), kThreads, 0, s>>>(boxes, m, kx.p, ky.p);
        RT_LAUNCH();
    }
    if (bits == 0)  // one slab: the y order is the packing order
        return radix_passes<END_VALUES>(ky.p, nullptr, k.p, pack, m, 0, 32, RadixEnd{END_VALUES, nullptr, 1}, s);
    RT_TRY(radix_passes<END_GROUPS>(kx.p, nullptr, k.p, v.p, m, 0, 32, RadixEnd{END_GROUPS, kx.p, size}, s));
    RT_TRY(radix_passes<END_RELABEL>(ky.p, nullptr, k.p, v.p, m, 0, 32, RadixEnd{END_RELABEL, kx.p, 1}, s));
    return radix_passes<END_VALUES>(k.p, v.p, ky.p, pack, m, 0, bits, RadixEnd{END_VALUES, nullptr, 1}, s);
}

// Levels up to this many boxes are packed by clusters: two sort
// the x and the y keys side by side, then one the y order by slab.  A tree
// of 20K boxes (F=16) builds in 270 us instead of 449, of 150K in 360 instead of
// 625, of 520K in 610 instead of 706; the sorts of a level use 32 SMs at most, so
// larger ones are left to the whole chip.
constexpr int64_t kLevelMost = (int64_t)1 << 19;

}  // namespace

rtree_status str_order(const float4 *boxes, int64_t m, int64_t size, uint32_t *pack, cudaStream_t s)
{
    int bits = 0;
    for (int64_t v = (m + size - 1) / size - 1; v; v >>= 1)
        ++bits;
    if (m > kLevelMost || cluster_ctas() == 0)
        return str_order_large(boxes, m, (uint32_t)size, bits, pack, s);
    DevBuf<uint32_t> buf(s);
    RT_TRY(buf.alloc(7 * (size_t)m, "level order"));
    uint32_t *x = buf.p, *y = x + 4 * m, *order_y = y + 2 * m;
    uint32_t *slab = x;  // the last x pass reads x + m and x + 3m
    // each sort ends in the first of its buffers; pack is one of the y sort's
    // on the way to order_y, or where it ends
    ClusterSort ax{nullptr, nullptr, boxes, nullptr, {x, x + m}, {x + 2 * m, x + 3 * m}, slab, (uint32_t)size,
                   0, (int)m, 0, 32, 4, 0};
    ClusterSort ay{nullptr, nullptr, boxes, nullptr, {y, y + m}, {bits ? order_y : pack, bits ? pack : order_y}, nullptr, 1,
                   1, (int)m, 0, 32, 4, 0};
    if (bits == 0)  // one slab: the y order is the packing order
        return launch_cluster<SRC_BOXES>(ay, ay, 1, s);
    RT_TRY(launch_cluster<SRC_BOXES>(ax, ay, 2, s));
    const ClusterSort as{nullptr, order_y, nullptr, slab, {y, y + m}, {pack, x + m}, nullptr, 1,
                         0, (int)m, 0, bits, (bits + 7) / 8, 0};
    return launch_cluster<SRC_TABLE>(as, as, 1, s);
}

}  // namespace rt
