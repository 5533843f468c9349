// join.cu -- R-tree join (Section 4), synchronized top-down traversal.
//
// Both trees are walked from their roots together (Brinkhoff, Kriegel and
// Seeger 1993): a node pair (a, b) whose entries intersect yields child
// pairs, and leaf pairs yield (r_id, s_id).  The frontier is processed one
// level at a time; every node pair is tested by one warp with the
// one-to-many comparison of Section 4.1: inner children sit one per lane,
// outer children's MBRs are broadcast to them, and __ballot_sync over the four
// comparisons gives the qualifying inner children, compacted with
// popc(mask & lanemask_lt) (queue insertion, step 4).  Children that miss the
// other node's bounding box are left out first.
// Where the heights differ, only the taller tree descends: its children are
// tested against the other node's bounding box.
//
// For trees whose node entries ascend by lx, equal-height pairs can use the
// prunings of Section 4.2 instead (k_join_pruned): O3 ends the outer loop at
// the first outer child whose lx lies right of every inner child, and O4/O5
// bound each outer child's inner scan by the number f of inner children that
// start left of its hx, found by the batched search of the many-to-many
// comparison.  The f candidate pairs of all lanes are then packed densely
// onto the warp, so a node pair costs ceil(sum f / 32) tests instead of one
// per outer child.
//
// A level is one pass: pairs are staged per warp and written through an atomic
// cursor (their order does not matter: the final (r_id, s_id) pairs are sorted
// lexicographically by two stable radix sorts, by s, then by r).
#include <algorithm>
#include <cstring>

#include "internal.cuh"

namespace rt {
namespace {

enum { J_BOTH = 0, J_A = 1, J_B = 2, J_LEAF = 3 };
enum { PASS_COUNT = 0, PASS_SCATTER = 1 };
constexpr int kThreads = 256;
constexpr uint32_t kSign = 0x80000000u;
constexpr int kMaxFanout = 128;

__device__ __forceinline__ float entry_lx(const TreeDev &t, int64_t g, int j)
{
    if (t.layout == RTREE_LAYOUT_AOS)
        return __ldg(reinterpret_cast<const float *>(t.mbr) + (g * t.fanout + j) * 4);
    if (t.layout == RTREE_LAYOUT_LOHI)
        return __ldg(t.mbr + g * 4 * t.fanout + 2 * j);
    return __ldg(t.mbr + g * 4 * t.fanout + j);
}

// Output of one level: pairs go to out[0 .. cap) through the counter *n,
// which keeps counting past cap (the level is then run again with room).
// bits (leaf level): OR and AND of the r ids, then of the s ids, for the sort.
struct JoinOut {
    int2 *out;
    unsigned long long *n;
    long long cap;
    uint32_t *bits;
};

// A warp's output on its way out: pairs are staged in shared memory and
// written with one reservation per kStage of them, so one pass over the node
// pairs is enough (a count pass before the writing pass was half the time)
// and the counter sees few atomics.
constexpr int kStage = 128;
struct WarpOut {
    const JoinOut &o;
    int2 *buf;
    int lane;
    unsigned lt;
    int n = 0;
    uint32_t r_or = 0, r_and = ~0u, s_or = 0, s_and = ~0u;
    __device__ __forceinline__ void flush()
    {
        if (n == 0)
            return;
        unsigned long long base = 0;
        if (lane == 0)
            base = atomicAdd(o.n, (unsigned long long)n);
        base = __shfl_sync(RT_FULL, base, 0);
        __syncwarp();
        for (int e = lane; e < n; e += 32)
            if ((long long)(base + e) < o.cap)
                o.out[base + e] = buf[e];
        __syncwarp();
        n = 0;
    }
    template <bool LEAF>
    __device__ __forceinline__ void emit(unsigned m, bool hit, int2 v)
    {
        if (n + __popc(m) > kStage)
            flush();
        if (hit) {
            buf[n + __popc(m & lt)] = v;
            if (LEAF) {
                r_or |= (uint32_t)v.x, r_and &= (uint32_t)v.x;
                s_or |= (uint32_t)v.y, s_and &= (uint32_t)v.y;
            }
        }
        n += __popc(m);
    }
    template <bool LEAF>
    __device__ __forceinline__ void finish()
    {
        flush();
        if (LEAF) {
            r_or = __reduce_or_sync(RT_FULL, r_or), r_and = __reduce_and_sync(RT_FULL, r_and);
            s_or = __reduce_or_sync(RT_FULL, s_or), s_and = __reduce_and_sync(RT_FULL, s_and);
            if (lane == 0) {
                atomicOr(o.bits, r_or);
                atomicAnd(o.bits + 1, r_and);
                atomicOr(o.bits + 2, s_or);
                atomicAnd(o.bits + 3, s_and);
            }
        }
    }
};

// Node pairs of one level: pairs[0 .. *np), or none if they did not all fit
// (the level before is run again).
__device__ __forceinline__ int64_t level_pairs(const unsigned long long *np, long long cap)
{
    const long long n = (long long)*np;
    return n <= cap ? n : 0;
}

// Candidates of a node: its children that meet `box`, compacted in order into
// shared memory.  Returns how many.
__device__ __forceinline__ int keep_meeting(const TreeDev &t, int g, int cnt, float4 box, float4 *kept,
                                            uint8_t *idx, int lane, unsigned lt)
{
    int n = 0;
    for (int i0 = 0; i0 < cnt; i0 += 32) {
        const int i = i0 + lane;
        const float4 e = i < cnt ? load_entry(t.mbr, t.layout, t.fanout, g, i) : empty_box();
        const bool ok = i < cnt && meets(e, box);
        const unsigned m = __ballot_sync(RT_FULL, ok);
        if (ok) {
            const int at = n + __popc(m & lt);
            kept[at] = e;
            idx[at] = (uint8_t)i;
        }
        n += __popc(m);
    }
    return n;
}

// Shared memory of a warp: the candidates of both nodes, and the staged output.
struct JoinWarp {
    float4 a[kMaxFanout], b[kMaxFanout];
    uint8_t ia[kMaxFanout], ib[kMaxFanout];
    int2 stage[kStage];
};
constexpr int kJoinWarps = 4;

// One warp per node pair (a, b), each taking every nwarps-th.
// Where both descend, only the children of a that meet b's bounding box and
// the children of b that meet a's can be in a qualifying pair (the
// search-space restriction of Brinkhoff, Kriegel and Seeger 1993).  On two
// leaves that touch that is about a third of either, so the one-to-many
// comparison of the survivors, packed onto the lanes (32/G outer ones a step
// for G inner ones), takes a few steps instead of one per outer child.
// Measured on the 2M x 2M join (F = 32, 273K node pairs, 989K results): all
// levels 0.21 ms, against 1.09 ms for a count and a writing pass that tested
// every outer child against all inner ones.  Bound by the latency of the
// nodes' loads and by issue.  Four warps a block: their shared memory (21 KB)
// and 64 registers leave 32 warps an SM.
template <int MODE>
__global__ void __launch_bounds__(32 * kJoinWarps)
    k_join(TreeDev ta, TreeDev tb, const int2 *__restrict__ pairs, const unsigned long long *__restrict__ np,
           long long np_cap, JoinOut jo)
{
    __shared__ JoinWarp smem[kJoinWarps];
    JoinWarp &sm = smem[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    const int64_t nwarps = (int64_t)gridDim.x * kJoinWarps;
    const int64_t count = level_pairs(np, np_cap);
    constexpr bool LEAF = MODE == J_LEAF;
    WarpOut w{jo, sm.stage, lane, lt};
    for (int64_t p = blockIdx.x * (int64_t)kJoinWarps + (threadIdx.x >> 5); p < count; p += nwarps) {
        const int2 pr = pairs[p];
        const int a = pr.x, b = pr.y;
        const int4 ma = __ldg(ta.meta + a), mb = __ldg(tb.meta + b);
        if (MODE == J_A) {
            const float4 bb = __ldg(tb.nbox + b);
            for (int i0 = 0; i0 < ma.y; i0 += 32) {
                const int i = i0 + lane;
                const bool hit = i < ma.y && meets(load_entry(ta.mbr, ta.layout, ta.fanout, a, i), bb);
                w.emit<false>(__ballot_sync(RT_FULL, hit), hit, make_int2(ma.x + i, b));
            }
        } else if (MODE == J_B) {
            const float4 ab = __ldg(ta.nbox + a);
            for (int j0 = 0; j0 < mb.y; j0 += 32) {
                const int j = j0 + lane;
                const bool hit = j < mb.y && meets(ab, load_entry(tb.mbr, tb.layout, tb.fanout, b, j));
                w.emit<false>(__ballot_sync(RT_FULL, hit), hit, make_int2(a, mb.x + j));
            }
        } else {
            const float4 ab = __ldg(ta.nbox + a), bb = __ldg(tb.nbox + b);
            __syncwarp();  // the previous pair's candidates are done with
            const int no = keep_meeting(ta, a, ma.y, bb, sm.a, sm.ia, lane, lt);
            const int ni = keep_meeting(tb, b, mb.y, ab, sm.b, sm.ib, lane, lt);
            __syncwarp();
            for (int j0 = 0; j0 < ni; j0 += 32) {
                const int left = ni - j0;
                const int lg = left > 16 ? 5 : left > 8 ? 4 : left > 4 ? 3 : 2;  // G = 2^lg inner ones
                const int j = j0 + (lane & ((1 << lg) - 1)), grp = lane >> lg;
                const bool vj = j < ni;
                const float4 eb = vj ? sm.b[j] : empty_box();
                for (int i0 = 0; i0 < no; i0 += 32 >> lg) {
                    const int i = i0 + grp;
                    const bool hit = vj && i < no && meets(sm.a[min(i, no - 1)], eb);
                    const unsigned m = __ballot_sync(RT_FULL, hit);
                    if (m) {
                        int2 v = make_int2(0, 0);
                        if (hit) {
                            v = make_int2(ma.x + sm.ia[i], mb.x + sm.ib[j]);
                            if (LEAF)
                                v = make_int2(__ldg(ta.ids + v.x), __ldg(tb.ids + v.y));
                        }
                        w.emit<LEAF>(m, hit, v);
                    }
                }
            }
        }
    }
    w.finish<LEAF>();
}

// Equal-height node pairs of two sorted-children trees, one pair per warp.
template <bool LEAF>
__global__ void __launch_bounds__(kThreads)
    k_join_pruned(TreeDev ta, TreeDev tb, const int2 *__restrict__ pairs, const unsigned long long *__restrict__ np,
                  long long np_cap, JoinOut jo)
{
    __shared__ float s_lx[kThreads / 32][kMaxFanout];
    __shared__ int2 s_stage[kThreads / 32][kStage];
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    float *lxs = s_lx[threadIdx.x >> 5];
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t count = level_pairs(np, np_cap);
    WarpOut w{jo, s_stage[threadIdx.x >> 5], lane, lt};
    for (int64_t p = warp; p < count; p += nwarps) {
        const int2 pr = pairs[p];
        const int a = pr.x, b = pr.y;
        const int4 ma = __ldg(ta.meta + a), mb = __ldg(tb.meta + b);
        const float4 bb = __ldg(tb.nbox + b);  // inner node MBR: max over children of hx is bb.z
        const int nin = mb.y;
        __syncwarp();  // the previous pair's searches are done with lxs
        for (int j = lane; j < nin; j += 32)
            lxs[j] = entry_lx(tb, b, j);
        __syncwarp();
        int P2 = 1, rounds = 1;  // inner count rounded up to a power of two; log2(P2)+1 rounds
        while (P2 < nin) {
            P2 <<= 1;
            ++rounds;
        }
        for (int i0 = 0; i0 < ma.y; i0 += 32) {
            const int i = i0 + lane;
            const bool vi = i < ma.y;
            const float4 ob = vi ? load_entry(ta.mbr, ta.layout, ta.fanout, a, i) : empty_box();
            const bool keyok = vi && ob.x <= bb.z;   // O3 key test against all inner children
            const bool cand = keyok && meets(ob, bb);  // search-space restriction
            int f = 0;
            if (cand) {  // O5: first inner index whose lx exceeds ob.hx
                int g = P2 >> 1, step = (P2 >> 2) > 1 ? (P2 >> 2) : 1;
                f = nin;
                for (int r = 0; r < rounds; ++r) {
                    const bool pass = g < nin && ob.z >= lxs[g];
                    if (!pass && g < f)
                        f = g;
                    g = pass ? g + step : g - step;
                    step = (step >> 1) > 1 ? (step >> 1) : 1;
                }
            }
            int incl = f;  // inclusive scan of the bounds over the lanes
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(RT_FULL, incl, o);
                if (lane >= o)
                    incl += u;
            }
            const int excl = incl - f;
            const int T = __shfl_sync(RT_FULL, incl, 31);
            for (int k0 = 0; k0 < T; k0 += 32) {
                const int k = k0 + lane;
                int own = 0;  // the lane whose run [excl, incl) holds k
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const int v = __shfl_sync(RT_FULL, incl, own + st - 1);
                    if (v <= k)
                        own += st;
                }
                const int ex = __shfl_sync(RT_FULL, excl, own);
                const float4 o = make_float4(__shfl_sync(RT_FULL, ob.x, own),
                                             __shfl_sync(RT_FULL, ob.y, own),
                                             __shfl_sync(RT_FULL, ob.z, own),
                                             __shfl_sync(RT_FULL, ob.w, own));
                const int j = k - ex;
                bool hit = false;
                if (k < T)
                    hit = meets(o, load_entry(tb.mbr, tb.layout, tb.fanout, b, j));
                const unsigned m = __ballot_sync(RT_FULL, hit);
                if (m) {
                    int2 v = make_int2(ma.x + i0 + own, mb.x + j);
                    if (LEAF && hit)
                        v = make_int2(__ldg(ta.ids + v.x), __ldg(tb.ids + v.y));
                    w.emit<LEAF>(m, hit, v);
                }
            }
            // O3: outer children ascend by lx, so after one fails the key test
            // every later one fails it too
            if (__ballot_sync(RT_FULL, vi && !keyok) != 0)
                break;
        }
    }
    w.finish<LEAF>();
}

// ------------------------------------------------ persistent queued form
// The same traversal with node pairs pulled from a device work queue
// instead of one launch per level: warps of a persistent grid take items
// (node pairs, one 64-bit word each) by ticket, test them with the
// one-to-many comparison, and publish the qualifying child pairs to new
// slots of the queue; leaf pairs yield (r_id, s_id).  `pending` counts items
// published but not finished; a warp waits for its ticket's slot to be
// filled or for pending to reach zero, which ends the pass.  Every wait is
// bounded (flag 4, reported as RTREE_ETIMEOUT).  Two passes over the same
// traversal: the count pass adds up the result pairs, the scatter pass
// writes them through an atomic cursor (the pairs are sorted afterwards).
enum { JQ_QUEUE_FULL = 1, JQ_OUT_FULL = 2, JQ_TIMEOUT = 4, JQ_MISMATCH = 8 };
constexpr unsigned long long kJEmpty = ~0ull;
constexpr long long kJoinWaitCycles = 2000000000LL;  // about one second
constexpr int kTickets = 4;  // queue slots a warp takes at once

// Level bases of one tree (node index where each level starts, root first).
struct Levels {
    int32_t base[RT_MAX_LEVELS];
    int32_t n;
};

struct JoinQueue {
    unsigned long long *items;
    long long cap;
    unsigned long long *head;
    unsigned long long *tail;
    long long *pending;
};

// Height of node g above the leaves (0 = leaf level).
__device__ __forceinline__ int height_of(const Levels &L, int g)
{
    int l = 0;
    for (int e = 1; e < L.n; ++e)
        if (g >= L.base[e])
            l = e;
    return L.n - 1 - l;
}

__device__ __forceinline__ unsigned long long pack_pair(int a, int b)
{
    return (unsigned long long)(unsigned)a | ((unsigned long long)(unsigned)b << 32);
}

// Per-warp staging of one item's output: child node pairs to publish and
// result pairs to write, flushed with one atomic reservation each, so that
// the queue's and the output's counters see few atomics per item.
struct JoinStage {
    unsigned long long push[kThreads / 32][kStage];
    int2 pairs[kThreads / 32][kStage];
};

// Publishes the np staged child pairs: pending is raised before the slots
// are reserved and written, so the pass cannot end while they are
// outstanding.
__device__ __forceinline__ void jq_flush_push(const JoinQueue &q, int32_t *flags, const unsigned long long *buf,
                                              int np, int lane)
{
    if (np == 0)
        return;
    unsigned long long pos = 0;
    if (lane == 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(q.pending), (unsigned long long)np);
        pos = atomicAdd(q.tail, (unsigned long long)np);
    }
    pos = __shfl_sync(RT_FULL, pos, 0);
    for (int e = lane; e < np; e += 32) {
        const unsigned long long at = pos + e;
        if ((long long)at < q.cap) {
            volatile unsigned long long *slot = q.items + at;
            *slot = buf[e];
        } else {  // dropped: the traversal is incomplete, the host redoes it by levels
            atomicOr(flags, JQ_QUEUE_FULL);
            atomicAdd(reinterpret_cast<unsigned long long *>(q.pending), ~0ull);
        }
    }
    __syncwarp();
}

__device__ __forceinline__ void jq_flush_pairs(unsigned long long *out_count, int2 *out, long long out_cap,
                                               int32_t *flags, const int2 *buf, int n, int lane)
{
    if (n == 0)
        return;
    unsigned long long base = 0;
    if (lane == 0)
        base = atomicAdd(out_count, (unsigned long long)n);
    base = __shfl_sync(RT_FULL, base, 0);
    for (int e = lane; e < n; e += 32) {
        if ((long long)(base + e) < out_cap)
            out[base + e] = buf[e];
        else
            atomicOr(flags, JQ_OUT_FULL);
    }
    __syncwarp();
}

// Emits one ballot round: result pairs (leaf) are counted (count pass) or
// staged for writing; child node pairs are staged for publishing.
template <int PASS>
__device__ __forceinline__ void jq_emit(const JoinQueue &q, unsigned long long *out_count, int2 *out,
                                        long long out_cap, int32_t *flags, unsigned m, bool hit, int2 v,
                                        bool leaf, int lane, unsigned lt, unsigned long long &leaf_cnt,
                                        unsigned long long *push, int &np, int2 *pbuf, int &npairs)
{
    const int n = __popc(m);
    if (n == 0)
        return;
    if (leaf) {
        if (PASS == PASS_COUNT) {
            leaf_cnt += n;
            return;
        }
        if (npairs + n > kStage) {
            jq_flush_pairs(out_count, out, out_cap, flags, pbuf, npairs, lane);
            npairs = 0;
        }
        if (hit)
            pbuf[npairs + __popc(m & lt)] = v;
        npairs += n;
        __syncwarp();
        return;
    }
    if (np + n > kStage) {
        jq_flush_push(q, flags, push, np, lane);
        np = 0;
    }
    if (hit)
        push[np + __popc(m & lt)] = pack_pair(v.x, v.y);
    np += n;
    __syncwarp();
}

template <int PASS, bool PRUNE>
__global__ void __launch_bounds__(kThreads)
    k_join_wq(TreeDev ta, TreeDev tb, Levels la, Levels lb, JoinQueue q, long long wait_cycles,
              unsigned long long *__restrict__ out_count, int2 *__restrict__ out, long long out_cap,
              int32_t *__restrict__ flags)
{
    __shared__ float s_lx[kThreads / 32][kMaxFanout];
    __shared__ JoinStage stage;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = lanemask_lt();
    float *lxs = s_lx[wid];
    unsigned long long *push = stage.push[wid];
    int2 *pbuf = stage.pairs[wid];
    const int Fa = ta.fanout, Fb = tb.fanout;
    unsigned long long warp_pairs = 0;  // count pass: result pairs found by this warp
    unsigned long long ticket = 0, ticket_end = 0;  // tickets are taken kTickets at a time
    for (;;) {
        if (ticket == ticket_end) {
            if (lane == 0)
                ticket = atomicAdd(q.head, (unsigned long long)kTickets);
            ticket = __shfl_sync(RT_FULL, ticket, 0);
            ticket_end = ticket + kTickets;
        }
        const unsigned long long my = ticket++;
        if ((long long)my >= q.cap)
            break;
        unsigned long long word = kJEmpty;
        if (lane == 0) {
            const long long t0 = clock64();
            const volatile unsigned long long *slot = q.items + my;
            const volatile long long *pend = q.pending;
            unsigned ns = 32;
            for (;;) {
                word = *slot;
                if (word != kJEmpty)
                    break;
                if (*pend == 0)
                    break;
                if (clock64() - t0 > wait_cycles) {
                    atomicOr(flags, JQ_TIMEOUT);
                    break;
                }
                __nanosleep(ns);
                if (ns < 2048)
                    ns <<= 1;
            }
            __threadfence();
        }
        word = __shfl_sync(RT_FULL, word, 0);
        if (word == kJEmpty)
            break;
        const int a = (int)(word & 0xffffffffull), b = (int)(word >> 32);
        const int ha = height_of(la, a), hb = height_of(lb, b);
        const int4 ma = __ldg(ta.meta + a), mb = __ldg(tb.meta + b);
        unsigned long long leaf_cnt = 0;
        int np = 0, npairs = 0;
        if (ha > hb) {  // only r descends
            const float4 bb = __ldg(tb.nbox + b);
            for (int i0 = 0; i0 < ma.y; i0 += 32) {
                const int i = i0 + lane;
                const bool hit = i < ma.y && meets(load_entry(ta.mbr, ta.layout, Fa, a, i), bb);
                const unsigned m = __ballot_sync(RT_FULL, hit);
                jq_emit<PASS>(q, out_count, out, out_cap, flags, m, hit, make_int2(ma.x + i, b), false, lane,
                              lt, leaf_cnt, push, np, pbuf, npairs);
            }
        } else if (hb > ha) {  // only s descends
            const float4 ab = __ldg(ta.nbox + a);
            for (int j0 = 0; j0 < mb.y; j0 += 32) {
                const int j = j0 + lane;
                const bool hit = j < mb.y && meets(ab, load_entry(tb.mbr, tb.layout, Fb, b, j));
                const unsigned m = __ballot_sync(RT_FULL, hit);
                jq_emit<PASS>(q, out_count, out, out_cap, flags, m, hit, make_int2(a, mb.x + j), false, lane,
                              lt, leaf_cnt, push, np, pbuf, npairs);
            }
        } else if (!PRUNE) {  // equal heights: one-to-many comparison
            const bool leaf = ha == 0;
            const int G = Fb < 32 ? Fb : 32;
            const int KO = 32 / G;
            const int grp = lane / G, sub = lane % G;
            for (int j0 = 0; j0 < mb.y; j0 += G) {
                const int j = j0 + sub;
                const bool vj = j < mb.y;
                const float4 ib = vj ? load_entry(tb.mbr, tb.layout, Fb, b, j) : empty_box();
                for (int i0 = 0; i0 < ma.y; i0 += KO) {
                    const int i = i0 + grp;
                    const bool vi = i < ma.y;
                    const float4 ob = vi ? load_entry(ta.mbr, ta.layout, Fa, a, i) : empty_box();
                    const bool hit = vi && vj && meets(ob, ib);
                    const unsigned m = __ballot_sync(RT_FULL, hit);
                    int2 v = make_int2(ma.x + i, mb.x + j);
                    if (leaf && hit && PASS == PASS_SCATTER)
                        v = make_int2(__ldg(ta.ids + ma.x + i), __ldg(tb.ids + mb.x + j));
                    jq_emit<PASS>(q, out_count, out, out_cap, flags, m, hit, v, leaf, lane, lt, leaf_cnt, push, np,
                                  pbuf, npairs);
                }
            }
        } else {  // equal heights of sorted trees: O3 and O5 as in k_join_pruned
            const bool leaf = ha == 0;
            const float4 bb = __ldg(tb.nbox + b);
            const int nin = mb.y;
            __syncwarp();
            for (int j = lane; j < nin; j += 32)
                lxs[j] = entry_lx(tb, b, j);
            __syncwarp();
            int P2 = 1, rounds = 1;
            while (P2 < nin) {
                P2 <<= 1;
                ++rounds;
            }
            for (int i0 = 0; i0 < ma.y; i0 += 32) {
                const int i = i0 + lane;
                const bool vi = i < ma.y;
                const float4 ob = vi ? load_entry(ta.mbr, ta.layout, Fa, a, i) : empty_box();
                const bool keyok = vi && ob.x <= bb.z;
                const bool cand = keyok && meets(ob, bb);
                int f = 0;
                if (cand) {
                    int g = P2 >> 1, step = (P2 >> 2) > 1 ? (P2 >> 2) : 1;
                    f = nin;
                    for (int r = 0; r < rounds; ++r) {
                        const bool pass = g < nin && ob.z >= lxs[g];
                        if (!pass && g < f)
                            f = g;
                        g = pass ? g + step : g - step;
                        step = (step >> 1) > 1 ? (step >> 1) : 1;
                    }
                }
                int incl = f;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(RT_FULL, incl, o);
                    if (lane >= o)
                        incl += u;
                }
                const int excl = incl - f;
                const int T = __shfl_sync(RT_FULL, incl, 31);
                for (int k0 = 0; k0 < T; k0 += 32) {
                    const int k = k0 + lane;
                    int own = 0;
#pragma unroll
                    for (int st = 16; st > 0; st >>= 1) {
                        const int v = __shfl_sync(RT_FULL, incl, own + st - 1);
                        if (v <= k)
                            own += st;
                    }
                    const int ex = __shfl_sync(RT_FULL, excl, own);
                    const float4 o = make_float4(__shfl_sync(RT_FULL, ob.x, own), __shfl_sync(RT_FULL, ob.y, own),
                                                 __shfl_sync(RT_FULL, ob.z, own), __shfl_sync(RT_FULL, ob.w, own));
                    const int j = k - ex;
                    bool hit = false;
                    if (k < T)
                        hit = meets(o, load_entry(tb.mbr, tb.layout, Fb, b, j));
                    const unsigned m = __ballot_sync(RT_FULL, hit);
                    const int io = i0 + own;
                    int2 v = make_int2(ma.x + io, mb.x + j);
                    if (leaf && hit && PASS == PASS_SCATTER)
                        v = make_int2(__ldg(ta.ids + ma.x + io), __ldg(tb.ids + mb.x + j));
                    jq_emit<PASS>(q, out_count, out, out_cap, flags, m, hit, v, leaf, lane, lt, leaf_cnt, push, np,
                                  pbuf, npairs);
                }
                if (__ballot_sync(RT_FULL, vi && !keyok) != 0)
                    break;
            }
        }
        warp_pairs += leaf_cnt;
        jq_flush_push(q, flags, push, np, lane);
        if (PASS == PASS_SCATTER)
            jq_flush_pairs(out_count, out, out_cap, flags, pbuf, npairs, lane);
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            atomicAdd(reinterpret_cast<unsigned long long *>(q.pending), ~0ull);  // -1: this item is done
        }
    }
    if (PASS == PASS_COUNT && lane == 0 && warp_pairs)
        atomicAdd(out_count, warp_pairs);
}

// Resets the queue to the one item (root, root) and zeroes the counter;
// hold adds items counted as pending but never published (0 in normal use).
__global__ void k_jq_init(unsigned long long *__restrict__ items, long long cap,
                          unsigned long long *__restrict__ ctl, unsigned long long *__restrict__ counter,
                          int hold)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < cap;
         i += (long long)gridDim.x * blockDim.x)
        items[i] = i == 0 ? pack_pair(0, 0) : kJEmpty;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl[0] = 0;  // head
        ctl[1] = 1;  // tail
        ctl[2] = 1 + hold;  // pending
        *counter = 0;
    }
}

__global__ void k_jq_check(const unsigned long long *__restrict__ cursor, const unsigned long long *__restrict__ want,
                           int32_t *__restrict__ flags)
{
    if (*cursor != *want)
        atomicOr(flags, JQ_MISMATCH);
}

using JoinKernel = void (*)(TreeDev, TreeDev, const int2 *, const unsigned long long *, long long, JoinOut);

JoinKernel pick(int mode, bool prune)
{
    switch (mode) {
    case J_BOTH: return prune ? k_join_pruned<false> : k_join<J_BOTH>;
    case J_A: return k_join<J_A>;
    case J_B: return k_join<J_B>;
    default: return prune ? k_join_pruned<true> : k_join<J_LEAF>;
    }
}

// The root pair and the counters of a join by levels: n[0] = 1 pair, the
// other levels' 0, the id bits empty.
__global__ void k_join_init(int2 *__restrict__ front, unsigned long long *__restrict__ n, int steps,
                            uint32_t *__restrict__ bits)
{
    if (threadIdx.x == 0)
        *front = make_int2(0, 0);
    for (int i = threadIdx.x; i <= steps; i += blockDim.x)
        n[i] = i == 0;
    if (threadIdx.x < 4)
        bits[threadIdx.x] = threadIdx.x & 1 ? 0xffffffffu : 0u;
}

__global__ void k_split_pairs(const int2 *__restrict__ p, int64_t n, uint32_t *__restrict__ key,
                              uint32_t *__restrict__ val)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int2 v = p[i];
        key[i] = (uint32_t)v.y ^ kSign;  // s first (least significant)
        val[i] = (uint32_t)v.x ^ kSign;  // the next sort's keys
    }
}

__global__ void k_merge_pairs(const uint32_t *__restrict__ r, const uint32_t *__restrict__ s,
                              int64_t n, int2 *__restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = make_int2((int)(r[i] ^ kSign), (int)(s[i] ^ kSign));
}

unsigned blocks_for(int64_t n)
{
    int64_t b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > 65536 ? 65536 : b));
}

// Highest bit + 1 in which ids differ, given their OR and AND.
int top_bit(uint32_t all_or, uint32_t all_and)
{
    int b = 0;
    for (uint32_t d = all_or ^ all_and; d; d >>= 1)
        ++b;
    return b;
}

// Sorts n (r, s) pairs lexicographically: stable sort by s, then by r, each on
// the low bits in which its ids differ.  `pairs` may have room to spare and is
// left with exactly n; it is given up in between, so that the sort holds 24
// bytes a pair at most.
rtree_status sort_pairs(DevBuf<int2> &pairs, int64_t n, int r_bits, int s_bits, cudaStream_t s)
{
    if (n <= 0)
        return pairs.alloc(0, "join pairs");
    DevBuf<uint32_t> k0(s), v0(s), k1(s), v1(s);
    RT_TRY(k0.alloc(n, "join sort"));
    RT_TRY(v0.alloc(n, "join sort"));
    {
        KernelTimer kt_("split_pairs", s);
        k_split_pairs<<<blocks_for(n), 256, 0, s>>>(pairs.p, n, k0.p, v0.p);
        RT_LAUNCH();
    }
    pairs.reset();
    RT_TRY(k1.alloc(n, "join sort"));
    RT_TRY(v1.alloc(n, "join sort"));
    RT_TRY(radix_sort_pairs(k0.p, v0.p, k1.p, v1.p, n, 0, s_bits, s));  // by s; v1 = r keys
    RT_TRY(radix_sort_pairs(v1.p, k1.p, v0.p, k0.p, n, 0, r_bits, s));  // by r; k0 = s keys
    k1.reset();
    v1.reset();
    RT_TRY(pairs.alloc(n, "join pairs"));
    {
        KernelTimer kt_("merge_pairs", s);
        k_merge_pairs<<<blocks_for(n), 256, 0, s>>>(v0.p, k0.p, n, pairs.p);
        RT_LAUNCH();
    }
    return RTREE_OK;
}

using JoinWqKernel = void (*)(TreeDev, TreeDev, Levels, Levels, JoinQueue, long long, unsigned long long *,
                              int2 *, long long, int32_t *);

Levels levels_of(const rtree *t)
{
    Levels L{};
    L.n = t->levels;
    for (int e = 0; e < t->levels; ++e)
        L.base[e] = (int32_t)t->level_base[e];
    return L;
}

}  // namespace

rtree_status tree_join_queue(const rtree *R, const rtree *S, bool prune, cudaStream_t s, rtree_result *res,
                             bool *redo_by_levels)
{
    *redo_by_levels = false;
    res->rows = 0;
    res->total = 0;
    res->offsets = nullptr;
    if (R->nodes == 0 || S->nodes == 0) {
        DevBuf<int32_t> ids(s);
        RT_TRY(ids.alloc(2, "join pairs"));
        res->ids = ids.release();
        return RTREE_OK;
    }
    const TreeDev ta = R->view(), tb = S->view();
    const Levels la = levels_of(R), lb = levels_of(S);
    const long long cap = std::max<long long>(1ll << 22, 8ll * (R->nodes + S->nodes));
    DevBuf<unsigned long long> items(s), ctl(s), counter(s);
    DevBuf<int32_t> flags(s);
    RT_TRY(items.alloc(cap, "join work queue"));
    RT_TRY(ctl.alloc(3, "join work queue counters"));
    RT_TRY(counter.alloc(2, "join pair counters"));  // [0] count pass total, [1] scatter cursor
    RT_TRY(flags.alloc(2, "join flags"));
    RT_CUDA(cudaMemsetAsync(flags.p, 0, 2 * sizeof(int32_t), s));
    const JoinQueue q{items.p, cap, ctl.p, ctl.p + 1, reinterpret_cast<long long *>(ctl.p + 2)};
    JoinWqKernel kc = prune ? k_join_wq<PASS_COUNT, true> : k_join_wq<PASS_COUNT, false>;
    JoinWqKernel ks = prune ? k_join_wq<PASS_SCATTER, true> : k_join_wq<PASS_SCATTER, false>;
    int per_sm = 0;
    RT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kc, kThreads, 0));
    const unsigned grid = (unsigned)((per_sm > 0 ? per_sm : 1) * sm_count());  // persistent: all resident
    const unsigned init_blocks = (unsigned)std::min<long long>((cap + 255) / 256, 65536);
    long long dbg_wait = 0;
    int dbg_hold = 0;
    debug_wq_take(&dbg_wait, &dbg_hold);
    {
        KernelTimer kt_("jq_init", s);
        k_jq_init<<<init_blocks, 256, 0, s>>>(items.p, cap, ctl.p, counter.p, dbg_hold ? 1 : 0);
        RT_LAUNCH();
    }
    {
        KernelTimer kt_(prune ? "join_pruned_queue_count" : "join_queue_count", s);
        kc<<<grid, kThreads, 0, s>>>(ta, tb, la, lb, q, dbg_wait > 0 ? dbg_wait : kJoinWaitCycles, counter.p,
                                     nullptr, 0, flags.p);
        RT_LAUNCH();
    }
    // the one host read: the number of pairs (it sizes the result) and the flags
    int64_t total = 0;
    {
        PostList pl{};
        pl.src[0] = counter.p;
        pl.words[0] = 2;
        pl.at[0] = 0;
        pl.src[1] = flags.p;
        pl.words[1] = 1;
        pl.at[1] = 2;
        pl.n = 2;
        uint32_t w[3];
        RT_TRY(read_words(pl, s, w, 3));
        total = (int64_t)((uint64_t)w[0] | ((uint64_t)w[1] << 32));
        if (w[2] & JQ_TIMEOUT)
            return fail(RTREE_ETIMEOUT, "join: a work-queue wait exceeded its limit");
        if (w[2] & JQ_QUEUE_FULL) {  // more node pairs than the queue holds
            *redo_by_levels = true;
            return RTREE_OK;
        }
        if (w[2])
            return fail(RTREE_EINTERNAL, "join count pass reported device flags 0x%x", w[2]);
    }
    if (total >= (int64_t)INT32_MAX)
        return fail(RTREE_EOVERFLOW, "join result of %lld pairs exceeds the 2^31-1 pairs the pair sort takes",
                    (long long)total);
    DevBuf<int2> pairs(s);
    RT_TRY(pairs.alloc(total, "join pairs"));
    {
        KernelTimer kt_("jq_init", s);
        k_jq_init<<<init_blocks, 256, 0, s>>>(items.p, cap, ctl.p, counter.p + 1, 0);
        RT_LAUNCH();
    }
    {
        KernelTimer kt_(prune ? "join_pruned_queue_scatter" : "join_queue_scatter", s);
        ks<<<grid, kThreads, 0, s>>>(ta, tb, la, lb, q, kJoinWaitCycles, counter.p + 1, pairs.p, total,
                                     flags.p);
        RT_LAUNCH();
    }
    {
        KernelTimer kt_("jq_check", s);
        k_jq_check<<<1, 1, 0, s>>>(counter.p + 1, counter.p, flags.p);
        RT_LAUNCH();
    }
    RT_TRY(sort_pairs(pairs, total, 32, 32, s));
    // the scatter pass and the sort run on in the order of s; their flags
    // reach the result's status
    RT_TRY(post_result_status(flags.p, s, res));
    res->total = total;
    res->ids = reinterpret_cast<int32_t *>(pairs.release());
    return RTREE_OK;
}

namespace {

// The join by levels of two trees that are not empty.  lean: no buffer is larger
// than what it is to hold (the levels are then run twice, first to count).
rtree_status join_levels(const rtree *R, const rtree *S, bool prune, bool lean, cudaStream_t s,
                         rtree_result *res, int64_t *stats)
{
    const TreeDev ta = R->view(), tb = S->view();
    // The modes of the levels are fixed by the heights alone.
    int mode[2 * RT_MAX_LEVELS], steps = 0;
    for (int ra = R->levels - 1, rb = S->levels - 1;; ++steps) {
        const int m = (ra == 0 && rb == 0) ? J_LEAF : ra > rb ? J_A : rb > ra ? J_B : J_BOTH;
        mode[steps] = m;
        if (m == J_LEAF)
            break;
        ra -= m != J_B;
        rb -= m != J_A;
    }
    ++steps;
    // All levels are enqueued at once, each reading the number of its node
    // pairs on the device; one host read at the end returns the counts.  The
    // buffers hold a few node pairs per node and a few results per rectangle;
    // a level that finds more says how many, and the traversal resumes at
    // that level with a buffer of that size.
    constexpr long long kMostPairs = 16ll << 20;
    const long long front_cap = lean ? 1 : std::min<long long>(8ll * (R->nodes + S->nodes) + 65536, kMostPairs);
    const long long out_cap = lean ? 1 : std::min<long long>(R->n + S->n + 65536, kMostPairs);
    DevBuf<int2> front[2] = {DevBuf<int2>(s), DevBuf<int2>(s)}, pairs(s);
    long long cap[3] = {front_cap, front_cap, out_cap};  // of front[0], front[1], pairs
    DevBuf<unsigned long long> n(s);
    DevBuf<uint32_t> bits(s);
    RT_TRY(front[0].alloc(front_cap, "join frontier"));
    RT_TRY(front[1].alloc(front_cap, "join frontier"));
    RT_TRY(pairs.alloc(out_cap, "join pairs"));
    RT_TRY(n.alloc(2 * RT_MAX_LEVELS + 1, "join counters"));
    RT_TRY(bits.alloc(4, "join id bits"));
    {
        KernelTimer kt_("join_init", s);
        k_join_init<<<1, 128, 0, s>>>(front[0].p, n.p, steps, bits.p);
        RT_LAUNCH();
    }
    uint64_t h[2 * RT_MAX_LEVELS + 1] = {};
    uint32_t hbits[4];
    for (int from = 0;;) {
        for (int e = from; e < steps; ++e) {
            const bool last = e == steps - 1;
            const int to = last ? 2 : (e + 1) & 1;
            const JoinOut jo{last ? pairs.p : front[to].p, n.p + e + 1, cap[to], bits.p};
            JoinKernel kern = pick(mode[e], prune);
            const bool pr = prune && (mode[e] == J_BOTH || mode[e] == J_LEAF);
            const int threads = pr ? kThreads : 32 * kJoinWarps;
            int per_sm = 0;
            RT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0));
            KernelTimer kt_(prune ? "join_pruned_levels" : "join_levels", s);
            kern<<<(unsigned)((per_sm > 0 ? per_sm : 1) * sm_count()), threads, 0, s>>>(
                ta, tb, front[e & 1].p, n.p + e, e == 0 ? 1 : cap[e & 1], jo);
            RT_LAUNCH();
        }
        {
            PostList pl{};
            pl.src[0] = n.p;
            pl.words[0] = 2 * (steps + 1);
            pl.at[0] = 0;
            pl.src[1] = bits.p;
            pl.words[1] = 4;
            pl.at[1] = 2 * (steps + 1);
            pl.n = 2;
            uint32_t w[2 * (2 * RT_MAX_LEVELS + 1) + 4];
            RT_TRY(read_words(pl, s, w, 2 * (steps + 1) + 4));
            memcpy(h, w, (steps + 1) * sizeof(uint64_t));
            memcpy(hbits, w + 2 * (steps + 1), sizeof(hbits));
        }
        int full = -1;  // the first level whose output did not fit
        for (int e = from; e < steps && full < 0; ++e)
            if ((long long)h[e + 1] > cap[e == steps - 1 ? 2 : (e + 1) & 1])
                full = e;
        if (full < 0)
            break;
        const int to = full == steps - 1 ? 2 : (full + 1) & 1;
        if (to == 2 && h[full + 1] >= (uint64_t)INT32_MAX)
            break;  // too many results for the sort: reported below
        DevBuf<int2> &buf = to == 2 ? pairs : front[to];
        if (to == 2)  // the last level needs its input only
            front[(full + 1) & 1].reset();
        cap[to] = (long long)h[full + 1];
        RT_TRY(buf.alloc(cap[to], to == 2 ? "join pairs" : "join frontier"));
        RT_CUDA(cudaMemsetAsync(n.p + full + 1, 0, (steps - full) * sizeof(unsigned long long), s));
        from = full;
    }
    const int64_t total = (int64_t)h[steps];
    if (stats) {
        std::fill_n(stats, 5, 0);
        for (int e = 0; e < steps; ++e)
            stats[mode[e]] += (int64_t)h[e];  // node pairs tested in this mode
        stats[4] = total;
    }
    if (total >= (int64_t)INT32_MAX)
        return fail(RTREE_EOVERFLOW, "join result of %lld pairs exceeds the 2^31-1 pairs the pair sort takes",
                    (long long)total);
    front[0].reset();
    front[1].reset();
    RT_TRY(sort_pairs(pairs, total, top_bit(hbits[0], hbits[1]), top_bit(hbits[2], hbits[3]), s));
    RT_CUDA(cudaStreamSynchronize(s));
    res->total = total;
    res->ids = reinterpret_cast<int32_t *>(pairs.release());
    return RTREE_OK;
}

}  // namespace

rtree_status tree_join(const rtree *R, const rtree *S, bool prune, cudaStream_t s,
                       rtree_result *res, int64_t *stats)
{
    res->rows = 0;
    res->total = 0;
    res->offsets = nullptr;
    if (R->nodes == 0 || S->nodes == 0) {
        DevBuf<int32_t> ids(s);
        RT_TRY(ids.alloc(2, "join pairs"));
        RT_CUDA(cudaStreamSynchronize(s));
        res->ids = ids.release();
        return RTREE_OK;
    }
    rtree_status st = join_levels(R, S, prune, false, s, res, stats);
    if (st == RTREE_ENOMEM) {  // once more without the room to spare
        clear_error();
        st = join_levels(R, S, prune, true, s, res, stats);
    }
    return st;
}

}  // namespace rt
