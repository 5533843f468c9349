// scan.cu -- exclusive prefix sums (reduce, scan of tile sums, scan tiles).
//
// Used for CSR offsets (per-query hit counts -> int64 offsets).  out has n+1
// entries; out[n] is the total, so one 8-byte read gives the output size.  Up to
// kScanJobs arrays of one length are scanned by the same launches.
#include "internal.cuh"

namespace rt {
namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T u = __shfl_up_sync(RT_FULL, v, d);
        if (lane >= d)
            v += u;
    }
    return v;
}

// Exclusive block scan of one value per thread; also returns the block total.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T &total)
{
    __shared__ T warp_tot[kThreads / 32];
    __shared__ T tot_sh;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31)
        warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        T t = lane < kThreads / 32 ? warp_tot[lane] : T(0);
        T ti = warp_incl_scan(t);
        if (lane < kThreads / 32)
            warp_tot[lane] = ti - t;
        if (lane == kThreads / 32 - 1)
            tot_sh = ti;
    }
    __syncthreads();
    total = tot_sh;
    T r = warp_tot[w] + inc - v;
    __syncthreads();  // the shared words may be reused by a later call
    return r;
}

// Notes a thread's largest value and the sum of those above j.over (ScanJobs::most).
__device__ __forceinline__ void note(int32_t *most, int32_t v, int64_t above)
{
    v = __reduce_max_sync(RT_FULL, v);
    if ((threadIdx.x & 31) == 0 && v > 0)
        atomicMax(most, v);
    if (above > 0)  // seldom
        atomicAdd(reinterpret_cast<unsigned long long *>(most + 2), (unsigned long long)above);
}

// The arrays of one launch (blockIdx.y): base, if given, is each tile's start.
template <typename Tin>
struct Scans {
    const Tin *in[kScanJobs];
    int64_t *out[kScanJobs];
    const int64_t *base[kScanJobs];
    int32_t *most[kScanJobs];
    int32_t over;
};

template <typename Tin>
__global__ void __launch_bounds__(kThreads) k_tile_reduce(const __grid_constant__ Scans<Tin> j, int64_t n)
{
    const Tin *__restrict__ in = j.in[blockIdx.y];
    const int64_t base = (int64_t)blockIdx.x * kTile;
    int64_t acc = 0, above = 0;
    Tin big = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        int64_t k = base + i * kThreads + threadIdx.x;
        if (k < n) {
            acc += (int64_t)in[k];
            big = in[k] > big ? in[k] : big;
            above += in[k] > j.over ? (int64_t)in[k] : 0;
        }
    }
    if (j.most[blockIdx.y])
        note(j.most[blockIdx.y], (int32_t)big, above);
    int64_t total;
    block_excl_scan<int64_t>(acc, total);
    if (threadIdx.x == 0)
        j.out[blockIdx.y][blockIdx.x] = total;
}

// Scans one tile; the last tile writes out[n] = total.
template <typename Tin>
__global__ void __launch_bounds__(kThreads) k_tile_scan(const __grid_constant__ Scans<Tin> j, int64_t n)
{
    __shared__ int64_t sm[kTile];
    const Tin *__restrict__ in = j.in[blockIdx.y];
    int64_t *__restrict__ out = j.out[blockIdx.y];
    const int64_t base = (int64_t)blockIdx.x * kTile;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        int p = i * kThreads + threadIdx.x;
        int64_t k = base + p;
        sm[p] = k < n ? (int64_t)in[k] : 0;
    }
    __syncthreads();
    int64_t v[kItems], run = 0, big = 0, above = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        v[i] = sm[threadIdx.x * kItems + i];
        run += v[i];
        big = v[i] > big ? v[i] : big;
        above += v[i] > j.over ? v[i] : 0;
    }
    if (j.most[blockIdx.y])
        note(j.most[blockIdx.y], (int32_t)big, above);
    int64_t total;
    int64_t pre = block_excl_scan<int64_t>(run, total);
    const int64_t tb = j.base[blockIdx.y] ? j.base[blockIdx.y][blockIdx.x] : 0;
    pre += tb;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        sm[threadIdx.x * kItems + i] = pre;
        pre += v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        int p = i * kThreads + threadIdx.x;
        int64_t k = base + p;
        if (k < n)
            out[k] = sm[p];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0)
        out[n] = tb + total;
}

// Arrays of one tile, one after another by one CTA, and then the words of l:
// a small call waits for the chain of its launches, and this is one for up to
// four (one query on 1M rectangles: 165 -> 153 us).
__global__ void __launch_bounds__(kThreads) k_scan_post(const __grid_constant__ ScanJobs j, int n,
                                                        const __grid_constant__ PostList l, uint32_t *__restrict__ dst)
{
    for (int a = 0; a < j.count; ++a) {
        const int32_t *__restrict__ in = j.in[a];
        const int k0 = threadIdx.x * kItems;
        int64_t v[kItems], run = 0, above = 0;
        int32_t big = 0;
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const int32_t x = k0 + i < n ? in[k0 + i] : 0;
            v[i] = run;
            run += x;
            big = x > big ? x : big;
            above += x > j.over ? x : 0;
        }
        if (j.most[a])
            note(j.most[a], big, above);
        int64_t total;
        const int64_t pre = block_excl_scan<int64_t>(run, total);
#pragma unroll
        for (int i = 0; i < kItems; ++i)
            if (k0 + i < n)
                j.out[a][k0 + i] = pre + v[i];
        if (threadIdx.x == 0)
            j.out[a][n] = total;
    }
    __threadfence();
    __syncthreads();
    const int i = threadIdx.x;
    if (i < l.n) {
        const volatile uint32_t *src = static_cast<const volatile uint32_t *>(l.src[i]);
        for (int w = 0; w < l.words[i]; ++w)
            dst[l.at[i] + w] = src[w];
    }
    mailbox_posted(dst);
}

template <typename Tin>
rtree_status scan_impl(const Scans<Tin> &j, int count, int64_t n, cudaStream_t s)
{
    const int64_t tiles = (n + kTile - 1) / kTile;
    if (tiles > INT32_MAX)
        return fail(RTREE_EOVERFLOW, "scan of %lld elements exceeds the grid limit", (long long)n);
    if (tiles == 1) {
        KernelTimer kt_("tile_scan", s);
        k_tile_scan<Tin><<<dim3(1, count), kThreads, 0, s>>>(j, n);
        RT_LAUNCH();
        return RTREE_OK;
    }
    DevBuf<int64_t> sums(s), sums_scan(s);
    RT_TRY(sums.alloc(count * tiles, "scan tile sums"));
    RT_TRY(sums_scan.alloc(count * (tiles + 1), "scan tile offsets"));
    Scans<Tin> reduce = j, scan = j;
    Scans<int64_t> up{};
    for (int a = 0; a < count; ++a) {
        reduce.out[a] = sums.p + a * tiles;
        up.in[a] = reduce.out[a];
        up.out[a] = sums_scan.p + a * (tiles + 1);
        scan.base[a] = up.out[a];
        scan.most[a] = nullptr;
    }
    {
        KernelTimer kt_("tile_reduce", s);
        k_tile_reduce<Tin><<<dim3((unsigned)tiles, count), kThreads, 0, s>>>(reduce, n);
        RT_LAUNCH();
    }
    RT_TRY(scan_impl<int64_t>(up, count, tiles, s));
    KernelTimer kt_("tile_scan", s);
    k_tile_scan<Tin><<<dim3((unsigned)tiles, count), kThreads, 0, s>>>(scan, n);
    RT_LAUNCH();
    return RTREE_OK;
}

}  // namespace

rtree_status scan_exclusive(const ScanJobs &j, int64_t n, cudaStream_t s)
{
    if (n <= 0) {
        for (int a = 0; a < j.count; ++a)
            RT_CUDA(cudaMemsetAsync(j.out[a], 0, sizeof(int64_t), s));
        return RTREE_OK;
    }
    Scans<int32_t> jobs{};
    for (int a = 0; a < j.count; ++a) {
        jobs.in[a] = j.in[a];
        jobs.out[a] = j.out[a];
        jobs.most[a] = j.most[a];
    }
    jobs.over = j.over;
    return scan_impl<int32_t>(jobs, j.count, n, s);
}

rtree_status scan_and_read(const ScanJobs &j, int64_t n, const PostList &l, cudaStream_t s, uint32_t *out, int nwords)
{
    if (n <= 0 || n > kTile) {
        RT_TRY(scan_exclusive(j, n, s));
        return read_words(l, s, out, nwords);
    }
    MailboxRef mb;
    RT_TRY(mailbox_get(&mb.m));
    mailbox_expect(mb.m);
    {
        KernelTimer kt_("scan_post", s);
        k_scan_post<<<1, kThreads, 0, s>>>(j, (int)n, l, mb.m.d);
        RT_LAUNCH();
    }
    return mailbox_take(mb.m, s, out, nwords);
}

}  // namespace rt
