// trig_kernels.cu -- sm_103a kernels of the online muon trigger (arXiv 1411.3968).
//
// Pipeline per batch of slices (all launches on one stream):
//   k_put      the batch's descriptors to the device, its counters zeroed.
//   k_bounds   structure pass of the k-way merge ("DAQ system": the Hit
//              Manager merges the PMT streams into time slices).  One read
//              of every hit: validates the CSR layout and ordering, and for
//              every tile g and PMT p records where p's stream crosses
//              the tile's halo edges B_g - H and B_{g+1} + H.
//   k_scatter  detectors above 128 PMTs: the hits copied to time buckets,
//              whose ranges then stand in for the PMT runs.
//   k_tile     persistent, warp-specialised: a stager warp dequeues tiles and
//              brings each tile's hits (one contiguous run per PMT) into
//              shared memory with bulk TMA copies (cp.async.bulk + mbarrier);
//              up to 16 consumer warps merge the runs into time order (bucket
//              sort on the time key), select seeds (charge threshold or
//              floor coincidence, "Sorting and triggering in GPU"), count
//              causally related hits per seed against the integer dt_max
//              table ("Muon trigger strategy"), and emit the fired seeds at
//              their merged rank.
//   k_final    stream compaction of the fired seeds, and the +-3 us windows
//              around the triggers, merged while lo_next <= hi_cur + 1, with
//              the hit count inside each: the difference of two merged ranks
//              the tile pass records beside each fired seed.
//
// Every wait on an mbarrier is bounded; a wait that gives up sets
// TRIG_FLAG_TIMEOUT on the batch and the kernel returns.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <cuda_runtime.h>

#include "trig_internal.h"

namespace trig {

// ------------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// try_wait with a suspend-time hint: a thread whose phase is not complete
// is suspended until it completes or about `ns` nanoseconds pass, instead
// of spinning and issuing instructions.
__device__ __forceinline__ bool mbar_try_wait_hint(uint64_t *bar, uint32_t parity, uint32_t ns)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity), "r"(ns)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Built with -DTRIG_PHASE_STATS, the tile kernel adds its per-phase clock
// cycles and its waits (cycles, try_wait rounds) into device counters that
// trig_phase_stats reads; without it the counters compile to nothing.
#ifdef TRIG_PHASE_STATS
__device__ unsigned long long g_phase[24];
#define PHASE_ADD(i, v) atomicAdd(&g_phase[(i)], (unsigned long long)(v))
#else
#define PHASE_ADD(i, v) ((void)0)
#endif
enum PhaseCounter {
    kPhTiles, kPhConsWait, kPhConsWaitRounds, kPhProdWait, kPhProdWaitRounds, kPhA, kPhB, kPhC, kPhD, kPhE,
    kPhF, kPhG, kPhSeeds, kPhProdItem, kPhConsTotal, kPhProdTotal, kPhKeys
};

// Bounded wait: gives up after limit_ns of the GPU's global timer and
// reports failure.  *rounds (optional) counts the try_wait rounds.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns,
                                          uint32_t *rounds = nullptr)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t_start = global_ns();
    for (uint32_t r = 1;; ++r) {
        if (rounds) *rounds = r;
        if (mbar_try_wait_hint(bar, parity, 20000u)) return true;
        if (global_ns() - t_start > limit_ns) return false;
    }
}

// Bulk (non-tensor) TMA copy global -> shared, completing on an mbarrier.
// Source and destination 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void named_sync(uint32_t id, uint32_t n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Named barrier over n threads that also ANDs a predicate across them: every
// thread leaves with the same answer.
__device__ __forceinline__ bool named_sync_and(uint32_t id, uint32_t n, bool p)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred q, o;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.and.pred o, %2, %3, q;\n\t"
        "selp.u32 %0, 1, 0, o;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v)
{
    const uint32_t lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (uint32_t)o) v += u;
    }
    return v;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ trig_hit load_hit(const trig_hit *p)
{
    int4 v = __ldg(reinterpret_cast<const int4 *>(p));
    trig_hit h;
    h.t_ns = (int64_t)(((uint64_t)(uint32_t)v.y << 32) | (uint32_t)v.x);
    h.pmt = (uint16_t)((uint32_t)v.z & 0xffffu);
    h.charge = (uint16_t)((uint32_t)v.z >> 16);
    h.reserved = (uint32_t)v.w;
    return h;
}

// first index i in [lo, hi) of a time-ordered hit run with t >= v
__device__ __forceinline__ uint64_t lb_time(const trig_hit *h, uint64_t lo, uint64_t hi, int64_t v)
{
    while (lo < hi) {
        uint64_t mid = lo + ((hi - lo) >> 1);
        if (h[mid].t_ns < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// --------------------------------------------------------------- self-check

// Built with -DTRIG_CHECK, every computed index into global or shared
// memory is checked first; a violation is recorded (the first one: site
// number, index, limit) and the access is skipped.  Without TRIG_CHECK the
// checks compile to nothing.
#ifdef TRIG_CHECK
struct CheckRecord {
    unsigned int site;
    unsigned int count;
    unsigned long long index, limit;
};
__device__ CheckRecord g_check;
__device__ __noinline__ bool check_fail(unsigned site, unsigned long long index, unsigned long long limit)
{
    if (atomicAdd(&g_check.count, 1u) == 0) {
        g_check.site = site;
        g_check.index = index;
        g_check.limit = limit;
    }
    return false;
}
#define CHECK(site, idx, lim) \
    (((unsigned long long)(idx) < (unsigned long long)(lim)) ? true : check_fail((site), (idx), (lim)))
#else
#define CHECK(site, idx, lim) true
#endif

// ------------------------------------------------------------------- dt_max

// Exact integer causality table.  For PMTs d mm apart the light needs
// d * n_num / (n_den * 1000) ns; dt_max = tol + ceil of that.  With
// X = n_num^2 * d^2 and r = floor(sqrt(X)): the ceiling is ceil(r / M) when
// X is a perfect square and floor(r / M) + 1 otherwise (M = n_den * 1000).
__global__ void k_dtmax(const int32_t *__restrict__ xyz, uint32_t P, uint32_t tol, uint32_t n_num,
                        uint32_t n_den, uint32_t corr, int32_t *__restrict__ dt_exact, uint16_t *__restrict__ dt)
{
    uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (uint64_t)P * P) return;
    uint32_t i = (uint32_t)(idx / P), j = (uint32_t)(idx % P);
    int64_t d2 = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int64_t dx = (int64_t)xyz[3 * i + c] - (int64_t)xyz[3 * j + c];
        d2 += dx * dx;
    }
    unsigned __int128 X = (unsigned __int128)((uint64_t)n_num * n_num) * (uint64_t)d2;
    uint64_t r = (uint64_t)sqrt((double)X);
    while ((unsigned __int128)r * r > X) --r;
    while ((unsigned __int128)(r + 1) * (r + 1) <= X) ++r;
    const uint64_t M = (uint64_t)n_den * 1000u;
    uint64_t k = ((unsigned __int128)r * r == X) ? (r + M - 1) / M : r / M + 1;
    uint64_t v = (uint64_t)tol + k;
    dt_exact[idx] = v > 0x7fffffffull ? 0x7fffffff : (int32_t)v;
    dt[idx] = (uint16_t)(v < corr ? v : corr);
}

__global__ void k_row_max(const uint16_t *__restrict__ dt, uint32_t P, uint16_t *__restrict__ dmax_row)
{
    uint32_t p = blockIdx.x;
    uint32_t m = 0;
    for (uint32_t q = threadIdx.x; q < P; q += blockDim.x) m = max(m, (uint32_t)dt[(size_t)p * P + q]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ uint32_t wm[32];
    if (lane_id() == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t r = 0;
        for (uint32_t w = 0; w < (blockDim.x + 31) / 32; ++w) r = max(r, wm[w]);
        dmax_row[p] = (uint16_t)r;
    }
}

cudaError_t launch_dtmax(const int32_t *xyz, uint32_t n_pmt, uint32_t tol, uint32_t n_num, uint32_t n_den,
                         uint32_t corr, int32_t *dt_exact, uint16_t *dt, uint16_t *dmax_row, cudaStream_t st)
{
    uint64_t n = (uint64_t)n_pmt * n_pmt;
    k_dtmax<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(xyz, n_pmt, tol, n_num, n_den, corr, dt_exact, dt);
    k_row_max<<<n_pmt, 256, 0, st>>>(dt, n_pmt, dmax_row);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ helpers

__device__ __forceinline__ uint32_t find_slice_by_item(const SliceDesc *desc, uint32_t n, uint32_t item)
{
    // largest s with desc[s].item0 <= item
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) >> 1;
        if (desc[mid].item0 <= item) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint32_t find_slice_by_chunk(const SliceDesc *desc, uint32_t n, uint32_t c)
{
    uint32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) >> 1;
        if (desc[mid].chunk0 <= c) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ void report(const SliceDesc &d, uint32_t flags)
{
    atomicOr(&d.stats->flags, flags);
}

// Time bucket of a wide slice: floor((t - O) / Wb) clamped to [0, NB).
// For offsets below 2^31 the high half of rel * ceil(2^32 / Wb) is the
// quotient or one more; one multiply corrects it.
__device__ __forceinline__ uint32_t bkt_index(const SliceDesc &d, int64_t t)
{
    const int64_t rel = t - d.bkt_origin;
    if (rel <= 0) return 0u;
    uint32_t q;
    if (d.bkt32 && rel < ((int64_t)1 << 31)) {
        const uint32_t r = (uint32_t)rel;
        q = __umulhi(r, d.bkt_magic);
        if (q * d.bkt_w > r) --q;
    } else {
        const int64_t q64 = rel / (int64_t)d.bkt_w;
        q = q64 >= (int64_t)d.n_bkt ? d.n_bkt : (uint32_t)q64;
    }
    return q < d.n_bkt ? q : d.n_bkt - 1;
}

// ---------------------------------------------------------------- k_bounds

__device__ __forceinline__ void fill_edges(uint32_t *e, uint32_t P, uint32_t p, uint32_t g0, uint32_t g1,
                                           uint32_t v)
{
    for (uint32_t g = g0; g < g1; ++g)
        if (CHECK(1, (size_t)g * P + p, (size_t)g1 * P)) e[(size_t)g * P + p] = v;
}

// The edges of the empty PMTs [q0, q1) before hit v of the slice (or past its
// last) are all v, if their offsets and that of q1 are; returns whether they
// are.  (No PMT has two places, so wrong offsets cost no more stores than
// right ones.)
__device__ __forceinline__ bool fill_empty(uint32_t *edge, const uint64_t *poff, uint32_t P, uint32_t NE, uint32_t q0,
                                           uint32_t q1, uint32_t v)
{
    for (uint32_t q = q0; q < q1; ++q) {
        if (poff[q] != v) return false;
        fill_edges(edge, P, q, 0, NE, v);
    }
    return poff[q1] == v;
}

constexpr int kBoundsThreads = 256;
constexpr int kBoundsUnroll = 4;
constexpr uint32_t kBoundsPerWarp = kChunkHits / (kBoundsThreads / 32);    // consecutive hits per warp
static_assert(kBoundsPerWarp == 31 * kBoundsUnroll, "a warp steps through 31 hits at a time");

// A slice's tile edges in time order.  Tile g's staged range starts at x = g W
// (its lo edge; x = t - (t0 - H)) and ends at g W + D, D = 2H + W = a W + b
// (its hi edge), so with x = q W + r the edges at or before x are
// 2 q + 1 + (r >= b): edge 2g is tile g's lo edge, edge 2 (g + a) + 1 its hi
// edge (the odd ones below 2a + 1 are no tile's).  One number per hit then
// tells both, and passing either kind of edge is the same store.
// A wide slice (WIDE) has the starts of its segments of buckets instead, one
// edge every edge_w ns.
template <bool WIDE>
struct EdgeCount {
    uint32_t W, magic, b, NE;
    __device__ __forceinline__ explicit EdgeCount(const SliceDesc &d)
        : W(d.edge_w), magic(d.w_magic), b(d.edge_b), NE(d.n_edges)
    {
    }
    // x below 2^31: the high half of x * ceil(2^32 / W) is the quotient or
    // one more
    __device__ __forceinline__ uint32_t of32(int32_t x) const
    {
        if (x < 0) return 0u;
        uint32_t q = __umulhi((uint32_t)x, magic);
        uint32_t r = (uint32_t)x - q * W;
        if ((int32_t)r < 0) --q, r += W;
        return min(WIDE ? q + 1u : 2u * q + (r >= b ? 2u : 1u), NE);
    }
    __device__ __forceinline__ uint32_t of64(int64_t x) const
    {
        if (x < 0) return 0u;
        const int64_t q = x / (int64_t)W;
        if (q >= (int64_t)(WIDE ? NE : NE / 2u)) return NE;
        return min(WIDE ? (uint32_t)q + 1u : 2u * (uint32_t)q + (x - q * (int64_t)W >= (int64_t)b ? 2u : 1u), NE);
    }
};

// Hit li of a slice where something other than a tile edge happens: the
// first or last hit of a PMT's run or of the slice, an out-of-range time, a
// step back.  It looks at the hit and its predecessor again (a run has
// thousands of hits, so few come here).
// A slice with hits that leaves here without a flag has its PMTs in order and
// every one of its P + 1 offsets at the place where that PMT's hits start:
// each run's first hit checks its own and those of the empty PMTs before it,
// the last hit those after it.  What follows takes offsets and edges as
// indices without a further look.
__device__ __noinline__ void bounds_special(const SliceDesc *dp, uint64_t li)
{
    const SliceDesc &d = *dp;
    const uint32_t P = d.n_pmt, NE = d.n_edges;
    const uint64_t *poff = d.pmt_off;
    const uint64_t n_hits = d.n_hits;
    const trig_hit h = load_hit(d.hits + li);
    trig_hit l = h;
    if (li > 0) l = load_hit(d.hits + li - 1);
    const uint32_t p = h.pmt, pl = l.pmt;
    const bool is_first = li == 0 || pl != p;
    uint32_t e, el;
    if (d.wide) {
        const EdgeCount<true> ec(d);
        e = ec.of64(h.t_ns - d.edge_org);
        el = ec.of64(l.t_ns - d.edge_org);
    } else {
        const EdgeCount<false> ec(d);
        e = ec.of64(h.t_ns - d.edge_org);
        el = ec.of64(l.t_ns - d.edge_org);
    }
    uint32_t bad = 0;
    if (p >= P || (li > 0 && pl > p)) bad |= TRIG_FLAG_BAD_PMT;
    else if (is_first) {
        if (!fill_empty(d.edge, poff, P, NE, li > 0 ? pl + 1u : 0u, p, (uint32_t)li)) bad |= TRIG_FLAG_BAD_PMT;
        else if (li > 0) fill_edges(d.edge, P, pl, el, NE, (uint32_t)li);       // hit li - 1 ended PMT pl's run
    }
    if (h.t_ns < d.in_lo || h.t_ns >= d.in_hi) bad |= TRIG_FLAG_OUT_OF_RANGE;
    if (!is_first && l.t_ns > h.t_ns) bad |= TRIG_FLAG_UNSORTED;
    if (bad) {
        report(d, bad);
        return;
    }
    fill_edges(d.edge, P, p, is_first ? 0u : el, e, (uint32_t)li);
    if (li + 1 == n_hits) {
        if (!fill_empty(d.edge, poff, P, NE, p + 1u, P, (uint32_t)n_hits)) report(d, TRIG_FLAG_BAD_PMT);
        else fill_edges(d.edge, P, p, e, NE, (uint32_t)n_hits);
    }
}

// Chunks [c, c_end) of one slice, block-wide.  A warp takes 31 new hits per
// step: lane 0 holds the hit before them, so every other lane's predecessor
// is its neighbour's and nothing is carried from step to step.  A lane whose
// hit has its predecessor's PMT and edge count, in order and in range, is
// done after that comparison; one that passes a tile edge writes its index.
// Bound by the latency of its loads and checks (issue 53 %, DRAM 51 %; nearly
// every step of 31 hits has a lane on the edge path, whose first store is
// predicated, the loop behind it rare): the 64 slices of both towers (205 M hits) take 0.91 ms, 1.42 with
// two edge counts per hit carried along walks of 512 hits (0.95 with a loop
// over the edges alone); one 320 k-hit slice 8 us, 13 before.  Four blocks an
// SM instead of three would spill: 254 against 210 us for 52 M hits.
template <bool WIDE, bool S32>
__device__ __forceinline__ void bounds_chunks(const SliceDesc &d, uint32_t c, uint32_t c_end)
{
    using T = std::conditional_t<S32, uint32_t, int64_t>;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, P = d.n_pmt;
    const uint32_t n_hits = (uint32_t)d.n_hits;                 // below 2^32 - 16
    const trig_hit *__restrict__ hits = d.hits;
    uint32_t *__restrict__ edge = d.edge;
    const int64_t in_lo = d.in_lo;
    const T in_span = (T)(d.in_hi - in_lo);
    const T x0 = (T)(d.edge_org - in_lo);                       // the first edge, from in_lo
    const EdgeCount<WIDE> ec(d);
    for (; c < c_end; ++c) {
        const uint32_t wbase = (c - d.chunk0) * kChunkHits + warp * kBoundsPerWarp;
        if (wbase >= n_hits) continue;
        uint4 v[kBoundsUnroll];
        uint32_t special = 0;
#pragma unroll
        for (int u = 0; u < kBoundsUnroll; ++u) {
            const uint32_t li = wbase + u * 31 + lane - 1u;      // wraps to 2^32 - 1 before the first hit
            v[u] = li < n_hits ? __ldg(reinterpret_cast<const uint4 *>(hits + li)) : make_uint4(0, 0, 0xffffu, 0);
        }
#pragma unroll
        for (int u = 0; u < kBoundsUnroll; ++u) {
            const uint32_t li = wbase + u * 31 + lane - 1u;
            const uint64_t rel = (((uint64_t)v[u].y << 32) | v[u].x) - (uint64_t)in_lo;
            const T r = (T)rel;
            const bool valid = li < n_hits, in = S32 ? (rel >> 32) == 0 && r < in_span : rel < (uint64_t)in_span;
            // PMT label; bits 16, 17: out of range, no such hit
            const uint32_t p = v[u].z & 0xffffu, pc = valid ? (in ? p : p | 0x10000u) : 0x2ffffu;
            uint32_t e = 0;
            if (in) e = S32 ? ec.of32((int32_t)(r - x0)) : ec.of64((int64_t)(r - x0));
            const uint32_t pcl = __shfl_up_sync(0xffffffffu, pc, 1);
            const T rl = __shfl_up_sync(0xffffffffu, r, 1);
            const uint32_t el = __shfl_up_sync(0xffffffffu, e, 1);
            if (lane == 0 || !valid) continue;
            if (pc != pcl || rl > r || !in || li + 1 == n_hits) special |= 1u << u;
            else if (e != el && p < P) {
                edge[(size_t)el * P + p] = li;          // most pass one edge at most
                if (e - el > 1u) fill_edges(edge, P, p, el + 1u, e, li);
            }
        }
        for (; special; special &= special - 1u)
            bounds_special(&d, wbase + (__ffs(special) - 1) * 31 + lane - 1u);
    }
}

// Slices longer than about two seconds, in 64-bit times.
__device__ __noinline__ void bounds_chunks_long(const SliceDesc &d, uint32_t c, uint32_t c_end)
{
    if (d.wide) bounds_chunks<true, false>(d, c, c_end);
    else bounds_chunks<false, false>(d, c, c_end);
}

// Structure pass: one read of every hit.  The CSR layout and the time order
// are checked (run starts and ends against pmt_off, each hit against its
// predecessor), and where each PMT's stream crosses the tile edges (wide
// slices: the edges of their segments of buckets) is recorded.  Each block takes a
// contiguous share of the chunks, so it looks its slice up once.
__global__ void __launch_bounds__(kBoundsThreads, 3) k_bounds(const BatchHeader *__restrict__ hdr,
                                                           const SliceDesc *__restrict__ desc)
{
    wait_for_previous_kernel();
    let_next_kernel_in();
    const uint32_t n_slices = hdr->n_slices, n_chunks = hdr->n_chunks;
    // no run of seeds is published yet (k_final)
    for (uint32_t i = blockIdx.x * kBoundsThreads + threadIdx.x; i < hdr->n_fin; i += gridDim.x * kBoundsThreads)
        *reinterpret_cast<uint32_t *>(hdr->fin + (size_t)i * kFinStateBytes) = 0;
    uint32_t c = (uint32_t)((uint64_t)n_chunks * blockIdx.x / gridDim.x);
    const uint32_t c1 = (uint32_t)((uint64_t)n_chunks * (blockIdx.x + 1) / gridDim.x);
    if (c >= c1) return;
    for (uint32_t s = find_slice_by_chunk(desc, n_slices, c); c < c1; ++s) {
        const SliceDesc &d = desc[s];
        const uint32_t end = min(c1, s + 1 < n_slices ? desc[s + 1].chunk0 : n_chunks);
        if (!d.span32) bounds_chunks_long(d, c, end);
        else if (d.wide) bounds_chunks<true, true>(d, c, end);
        else bounds_chunks<false, true>(d, c, end);
        c = end;
    }
}

// --------------------------------------------------------------- k_scatter

// Wide slices: every hit copied to its time bucket's range of tbuf (the
// order inside a bucket is arbitrary; the tile pass sorts), and the buckets'
// offsets.  A block takes one segment of seg_bkt buckets at a time: it reads
// each PMT's run in the segment (eight hits on average, sixteen lanes a run),
// counts them per bucket in shared memory, scans the counts from the
// segment's merged rank (the sum of the runs' places), and reads the runs
// again, from L2, to write them.  The writes of a block land in one window
// of tbuf (8 P hits), so L2 fills whole lines; the global counters that a
// hit-by-hit copy needs took 0.51 ms for the 2688-PMT slice (29.6 M hits)
// and 0.24 of the structure pass, against 0.42 and 0.13.  Bound by the
// latency of the short runs' loads.
// Slices with malformed input (flagged by the structure pass) are skipped, and
// so are those without hits, whose edges the structure pass never writes.
constexpr uint32_t kScatThreads = 512;

__global__ void __launch_bounds__(kScatThreads, 2) k_scatter(const BatchHeader *__restrict__ hdr,
                                                          const SliceDesc *__restrict__ desc)
{
    constexpr uint32_t NW = kScatThreads / 32;
    __shared__ uint32_t cnt[kSegBuckets], red[NW + 1];
    wait_for_previous_kernel();
    let_next_kernel_in();
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    for (uint32_t s = 0; s < hdr->n_slices; ++s) {
        const SliceDesc &d = desc[s];
        if (!d.wide || d.n_hits == 0) continue;
        if (d.stats->flags & (TRIG_FLAG_BAD_PMT | TRIG_FLAG_UNSORTED | TRIG_FLAG_OUT_OF_RANGE)) continue;
        const uint32_t P = d.n_pmt, K = d.seg_bkt, n_seg = d.n_edges - 1u;
        for (uint32_t g = blockIdx.x; g < n_seg; g += gridDim.x) {
            const uint32_t *ea = d.edge + (size_t)g * P, *eb = ea + P;
            const uint32_t b0 = g * K, nb = min(K, d.n_bkt - b0);
            const int64_t org = d.bkt_origin + (int64_t)b0 * d.bkt_w;
            for (uint32_t b = tid; b < nb; b += kScatThreads) cnt[b] = 0;
            __syncthreads();
            // bucket in the segment; a segment is shorter than 2^31 ns
            auto bucket = [&](const int4 &v) {
                const uint32_t rel = (uint32_t)((((uint64_t)(uint32_t)v.y << 32) | (uint32_t)v.x) - (uint64_t)org);
                uint32_t q = __umulhi(rel, d.bkt_magic);
                if (q * d.bkt_w > rel) --q;
                return min(q, nb - 1u);
            };
            // each half warp takes four runs at a time, their loads in flight
            // together
            auto each = [&](auto &&f) {
                for (uint32_t p0 = 2u * warp + (lane >> 4); p0 < P; p0 += 8u * NW) {
                    uint32_t i[4], e[4];
                    int4 v[4];
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u) {
                        const uint32_t p = p0 + u * 2u * NW;
                        i[u] = p < P ? ea[p] + (lane & 15u) : 0u;
                        e[u] = p < P ? eb[p] : 0u;
                    }
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u)
                        if (i[u] < e[u]) v[u] = *reinterpret_cast<const int4 *>(d.hits + i[u]);
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u) {
                        if (i[u] < e[u]) f(v[u]);
                        for (uint32_t k = i[u] + 16u; k < e[u]; k += 16u) f(*reinterpret_cast<const int4 *>(d.hits + k));
                    }
                }
            };
            each([&](const int4 &v) { atomicAdd(&cnt[bucket(v)], 1u); });
            // merged rank of the segment's first hit
            uint32_t base = 0;
            for (uint32_t p = tid; p < P; p += kScatThreads) base += ea[p] - (uint32_t)d.pmt_off[p];
            base = __reduce_add_sync(0xffffffffu, base);
            if (lane == 0) red[warp] = base;
            __syncthreads();
            base = __reduce_add_sync(0xffffffffu, lane < NW ? red[lane] : 0u);
            __syncthreads();
            // exclusive scan of the counts, kSegBuckets / threads each
            constexpr uint32_t V = kSegBuckets / kScatThreads;
            uint32_t v[V], own = 0;
#pragma unroll
            for (uint32_t i = 0; i < V; ++i) {
                v[i] = tid * V + i < nb ? cnt[tid * V + i] : 0u;
                own += v[i];
            }
            const uint32_t incl = warp_incl_scan(own);
            if (lane == 31) red[warp] = incl;
            __syncthreads();
            uint32_t run = base + __reduce_add_sync(0xffffffffu, lane < warp ? red[lane % NW] : 0u) + incl - own;
#pragma unroll
            for (uint32_t i = 0; i < V; ++i) {
                const uint32_t b = tid * V + i;
                if (b < nb) {
                    cnt[b] = run;
                    d.bkt_off[b0 + b] = run;
                }
                run += v[i];
            }
            if (g + 1 == n_seg && tid == kScatThreads - 1) d.bkt_off[d.n_bkt] = run;
            __syncthreads();
            each([&](const int4 &v) {
                const uint32_t pos = atomicAdd(&cnt[bucket(v)], 1u);
                if (CHECK(17, pos, d.n_hits)) *reinterpret_cast<int4 *>(d.tbuf + pos) = v;
            });
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ k_tile

struct ItemInfo {
    int32_t item;       // -1: no more work
    uint32_t slice;
    uint32_t g;
    uint32_t n;         // staged hits
    uint32_t rank_lo;   // merged rank of the first staged hit
    uint32_t mode;      // kItem*
    uint32_t off;       // start of the core, from the tile's (ns)
    uint32_t core;      // length of the core
    uint32_t lo_t;      // start of the core, from the staged range's
    uint32_t span;      // length of the staged range
};
// A whole staged tile; nothing to do (bad slice or empty); a staged piece of a
// tile, and the end of a tile's pieces; a tile put off until the block has no
// others, for tile_overflow (what was done of its pieces is dropped).
enum : uint32_t { kItemTile, kItemSkip, kItemPiece, kItemEnd, kItemDefer };

// Shared memory of the tile kernel, in this order: the staging buffer (handed
// back after its first read, so the next tile's copy overlaps the rest of the
// pass); the keys in bucket order (+16 bytes of end keys that the causal
// count's 16-byte loads may read past the last key); the floor cells, two
// bits each, whose place the seed list takes; the candidate list (position
// and charge), whose place the seeds' counts and the fired seeds' charges by
// position take; the bucket offsets; the
// mask of fired positions; the extended builds' (EXT) charges in key order
// and, for detectors above 128 PMTs, a 4096-bit PMT set per warp; the dt rows
// (kDtRow bytes each, 256-byte aligned) when the detector's table fits
// (NARROW); the PMT tables (floor, row maximum of dt).
// CROWD: the layout of crowd_pass, which takes twice the hits in the same
// memory: no staging buffer (its records, 8 bytes each, lie where the keys and
// candidates come later), half as many buckets and cells for a hit; the PMT
// sets and tables stay where they are.
template <int CAP, int NC, bool NARROW, bool EXT, bool CROWD = false>
struct TileLayout {
    static constexpr int NBK = CROWD ? CAP / 2 : CAP;      // time buckets
    static constexpr uint32_t kCells = 16u * NBK;          // floor cells
    static constexpr size_t kStage = CROWD ? 0 : (size_t)CAP * 16;
    static constexpr size_t oPk = kStage;
    static constexpr size_t kLists = (size_t)CAP * 4;      // the cells (or seeds), and the candidates
    static constexpr size_t oCell = oPk + (size_t)CAP * 4 + 16 + (CROWD ? kLists : 0);
    static constexpr size_t oCand = CROWD ? oPk + (size_t)CAP * 4 + 16 : oCell + kLists;
    static constexpr size_t oCnt = oPk + (size_t)CAP * 4 + 16 + 2 * kLists;
    static constexpr size_t oMask = oCnt + (size_t)(NBK + 1) * 4;
    static_assert(kCells / 4 <= kLists, "the cells and the seed list share their place");
    static constexpr size_t oChg = oMask + (size_t)(CAP / 32) * 4;
    static constexpr size_t oEnd = oChg + (EXT ? (size_t)CAP * 2 : 0);
    static constexpr size_t tables(size_t set) { return (set + (EXT && !NARROW ? (size_t)NC / 32 * 512 : 0) + kDtRow - 1) & ~(size_t)(kDtRow - 1); }
    static constexpr size_t oSet = CROWD ? TileLayout<CAP / (CROWD ? 2 : 1), NC, NARROW, EXT, false>::oSet : oEnd;
    static constexpr size_t oDt = tables(oSet);
    static_assert(oEnd <= oSet, "fits below what it leaves in place");
    static_assert(oCnt % 16 == 0 && oCell % 16 == 0, "cleared and scanned as 16-byte vectors");
    __host__ __device__ static size_t tab(uint32_t P) { return oDt + (NARROW ? (size_t)P * kDtRow : 0); }
    static size_t bytes(uint32_t P) { return (tab(P) + 2 * (size_t)((P + 7) & ~7u) * 2 + 127) & ~(size_t)127; }
};

// Dynamic shared memory of the tile kernel (layout TileLayout).
extern __shared__ __align__(256) unsigned char g_tile_smem[];

// The tile kernel's shared-memory regions sit at fixed offsets, so their
// addresses are recomputed where used instead of living in registers through
// every phase; only the PMT tables' place depends on the launch.  NARROW: at
// most kSmemDtMaxPmt PMTs in the batch and every dt table in shared memory.
template <int CAP, int NC, bool NARROW, bool EXT, bool CROWD = false>
struct TileCtx {
    using L = TileLayout<CAP, NC, NARROW, EXT, CROWD>;
    uint32_t P;             // PMTs of the loaded slice
    uint32_t tab;           // offset of the PMT tables
    uint32_t pp;            // their stride
    const uint16_t *dt_g;   // the loaded slice's dt table in global memory
    __device__ __forceinline__ uint64_t *stage() const { return reinterpret_cast<uint64_t *>(g_tile_smem); }
    __device__ __forceinline__ uint32_t *pk() const { return reinterpret_cast<uint32_t *>(g_tile_smem + L::oPk); }
    __device__ __forceinline__ uint32_t *seeds() const { return reinterpret_cast<uint32_t *>(g_tile_smem + L::oCell); }
    __device__ __forceinline__ uint32_t *cand() const { return reinterpret_cast<uint32_t *>(g_tile_smem + L::oCand); }
    __device__ __forceinline__ uint16_t *counts() const { return reinterpret_cast<uint16_t *>(g_tile_smem + L::oCand); }
    // a fired seed's charge at its position (the extended builds have every key's)
    __device__ __forceinline__ uint16_t *fired_charge() const { return EXT ? chg() : counts() + CAP; }
    __device__ __forceinline__ uint32_t *cnt() const { return reinterpret_cast<uint32_t *>(g_tile_smem + L::oCnt); }
    __device__ __forceinline__ uint32_t *cells() const { return reinterpret_cast<uint32_t *>(g_tile_smem + L::oCell); }
    __device__ __forceinline__ uint32_t *mask() const { return reinterpret_cast<uint32_t *>(g_tile_smem + L::oMask); }
    // the extended builds' charges, and warp w's PMT set
    __device__ __forceinline__ uint16_t *chg() const { return reinterpret_cast<uint16_t *>(g_tile_smem + L::oChg); }
    __device__ __forceinline__ uint32_t *pmt_set(uint32_t w) const
    {
        return reinterpret_cast<uint32_t *>(g_tile_smem + L::oSet) + 128 * w;
    }
    __device__ __forceinline__ uint16_t *dt_s() const { return reinterpret_cast<uint16_t *>(g_tile_smem + L::oDt); }
    __device__ __forceinline__ uint16_t *floor_s() const { return reinterpret_cast<uint16_t *>(g_tile_smem + tab); }
    __device__ __forceinline__ uint16_t *dmax_s() const { return floor_s() + pp; }
    // Packed key: time within the staged range (below 2^20 ns) above the PMT.
    // With at most 128 PMTs the PMT is kept doubled in eight bits, its byte
    // offset in a dt row; else in twelve bits.
    static constexpr uint32_t kShift = NARROW ? 8 : 12;
    static constexpr uint32_t kPmtMask = (1u << kShift) - 1u;
    static __device__ __forceinline__ uint32_t key(uint32_t t, uint32_t pmt)
    {
        return (t << kShift) | (NARROW ? pmt << 1 : pmt);
    }
    // dt entry of a row (seed rule 1 keeps the PMT relation in its upper bits)
    struct Row {
        uint32_t s;
        const uint16_t *g;
        __device__ __forceinline__ uint32_t at(uint32_t k) const
        {
            if (NARROW) return *reinterpret_cast<const uint16_t *>(g_tile_smem + (s | (k & kPmtMask)));
            return __ldg(g + key_p(k));
        }
    };
    __device__ __forceinline__ Row row(uint32_t p) const
    {
        return Row{(uint32_t)L::oDt + p * kDtRow, dt_g + (size_t)p * P};
    }
    static __device__ __forceinline__ uint32_t key_t(uint32_t k) { return k >> kShift; }
    static __device__ __forceinline__ uint32_t key_p(uint32_t k) { return NARROW ? (k & kPmtMask) >> 1 : k & kPmtMask; }
};

constexpr uint32_t kBarCons = 1;        // named barrier of the consumers

template <int NC>
__device__ __forceinline__ void cons_sync() { named_sync(kBarCons, NC); }

constexpr uint32_t kPkNone = 0xffffffffu;       // "no hit", above every key
constexpr uint32_t kNoItem = 0xffffffffu;       // end of the list of tiles put off

// Bucket of a time relative to the tile base: t_rel >> bsh, the last of
// the NB buckets taking everything beyond.
template <uint32_t NB>
__device__ __forceinline__ uint32_t bucket_of(uint32_t t_rel, uint32_t bsh)
{
    const uint32_t b = t_rel >> bsh;
    return b < NB ? b : NB - 1;
}

struct CoreOut {
    uint32_t n_fired;
    uint32_t n_seeds;
    uint32_t c0;
};

// The loaded slice's trigger parameters.
struct TrigParams {
    uint32_t H, tau, q_seed, threshold, win_half;
    uint32_t l0_hits, l0_window, l0_distinct;
    uint32_t seed_rule, sc_w, fc_w, afc_w, count_distinct;
    uint32_t dt_mask;       // the dt bits of a shared-memory row's entry
    const uint8_t *rel;
    trig_hit *dbg_merged;
    uint32_t *dbg_seedcnt;
};

// Seed rule 1 for the key at position i: [SC and AFC] or [FC and AFC].  Looks
// through the buckets of the widest of the three windows, four keys at a
// time (all staged: the tile halo covers it), and each pair up in the PMT
// relation row of p_i: the upper bits of the dt row where they hold it, else
// the table in global memory.
template <uint32_t NB, class CTX>
__device__ __forceinline__ bool coincidence_seed(const CTX &cx, const TrigParams &tp, uint32_t i, uint32_t bsh)
{
    const uint32_t *pk = cx.pk(), *cnt = cx.cnt();
    const uint32_t ki = pk[i], ti = CTX::key_t(ki), pi = CTX::key_p(ki);
    if (!CHECK(14, pi, cx.P)) return false;
    const uint8_t *rel = tp.rel + (size_t)pi * cx.P;
    const auto row = cx.row(pi);
    const bool packed = tp.dt_mask != 0xffffu;
    const uint32_t sc = tp.sc_w, fc = tp.fc_w, afc = tp.afc_w, w = max(sc, max(fc, afc));
    uint32_t j = cnt[(ti > w ? ti - w : 0u) >> bsh];
    const uint32_t je = cnt[bucket_of<NB>(ti + w, bsh) + 1];
    bool c = false, a = false;
    for (; j < je && !(a && c); j += 4) {
        uint32_t kj[4], r[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) kj[u] = pk[min(j + u, je - 1u)];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) r[u] = packed ? row.at(kj[u]) >> kRelShift : __ldg(rel + CTX::key_p(kj[u]));
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t d = __usad(CTX::key_t(kj[u]), ti, 0u);
            c = c || ((r[u] & kRelAdjacent) && d <= sc) || ((r[u] & kRelFloor) && d <= fc);
            a = a || ((r[u] & kRelNextFloor) && d <= afc);
        }
    }
    return a && c;
}

// A seed's scan range: the keys [j0, j1) of the buckets covering
// [t_s - d, t_s + d], d its row's maximum (keys beyond fail the causal
// test), from the sorted tile's bucket offsets.
template <uint32_t NB, class CTX>
__device__ __forceinline__ void seed_range(const CTX &cx, uint32_t ts, uint32_t ps, uint32_t bsh,
                                           uint32_t &j0, uint32_t &j1)
{
    const uint32_t dm = ps < cx.P ? (uint32_t)cx.dmax_s()[ps] : 0u;
    const uint32_t *boff = cx.cnt();
    j0 = boff[bucket_of<NB>(ts >= dm ? ts - dm : 0u, bsh)];
    j1 = boff[bucket_of<NB>(ts + dm, bsh) + 1];
}

// Distinct-PMT causal count: c(s) = the number of different PMTs among the
// keys j with |t_j - t_s| <= min(dt_max[p_s][p_j], W).  Up to 128 PMTs,
// eight lanes per seed each collect a 128-bit PMT set in registers over four
// consecutive keys at a time of the seed's scan range (keys outside it fail
// the test, see count_seeds), and the sets are OR-ed and counted; above, a
// warp per seed marks the PMTs in a shared-memory set.
template <uint32_t NB, int NC, class CTX>
__device__ __forceinline__ void count_distinct_pmts(const CTX &cx, uint32_t n, uint32_t ns, uint32_t bsh, uint32_t threshold,
                                                    uint32_t dt_mask)
{
    constexpr uint32_t G = 8, NG = NC / G;
    const uint32_t tid = threadIdx.x, gl = tid & (G - 1u), gid = tid / G, P = cx.P;
    const uint32_t *pk = cx.pk(), *seeds = cx.seeds();
    auto done = [&](uint32_t k, uint32_t pos, uint32_t c) {
        cx.counts()[k] = (uint16_t)c;
        if (c >= threshold) atomicOr(&cx.mask()[pos >> 5], 1u << (pos & 31u));
    };
    if (P > 128) {
        const uint32_t warp = tid >> 5, lane = tid & 31u, nwords = (P + 31u) >> 5;
        uint32_t *set = cx.pmt_set(warp);
        for (uint32_t k = warp; k < ns; k += NC / 32) {
            for (uint32_t w = lane; w < nwords; w += 32) set[w] = 0u;
            __syncwarp();
            const uint32_t pos = seeds[k] & 0xffffu, ks = pk[pos];
            const uint32_t ts = CTX::key_t(ks), ps = CTX::key_p(ks);
            uint32_t j0, j1;
            seed_range<NB>(cx, ts, ps, bsh, j0, j1);
            if (CHECK(12, j1, n + 1) && CHECK(13, ps, P) && CHECK(16, nwords, 129)) {
                const auto row = cx.row(ps);
                for (uint32_t q = j0 + lane; q < j1; q += 32) {
                    const uint32_t kj = pk[q], tj = CTX::key_t(kj), pj = CTX::key_p(kj);
                    if (!CHECK(11, pj, P)) continue;
                    if (__usad(tj, ts, 0u) <= row.at(kj)) atomicOr(&set[pj >> 5], 1u << (pj & 31u));
                }
            }
            __syncwarp();
            uint32_t c = 0;
            for (uint32_t w = lane; w < nwords; w += 32) c += __popc(set[w]);
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) done(k, pos, c);
            __syncwarp();                       // the set is read before the next seed clears it
        }
        return;
    }
    const uint32_t rounds = (ns + NG - 1) / NG;
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t k = r * NG + gid;
        uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0, pos = 0;
        if (k < ns) {
            pos = seeds[k] & 0xffffu;
            const uint32_t ks = pk[pos], ts = CTX::key_t(ks), ps = CTX::key_p(ks);
            uint32_t j0, j1;
            seed_range<NB>(cx, ts, ps, bsh, j0, j1);
            if (CHECK(12, j1, n + 1) && CHECK(13, ps, P)) {
                const auto row = cx.row(ps);
                auto mark = [&](uint32_t kj) {
                    const uint32_t pj = CTX::key_p(kj);
                    if (!CHECK(11, pj, P)) return;
                    const bool in = __usad(CTX::key_t(kj), ts, 0u) <= (row.at(kj) & dt_mask);
                    const uint32_t b = in ? 1u << (pj & 31u) : 0u, h = pj >> 5;
                    m0 |= h == 0 ? b : 0u;
                    m1 |= h == 1 ? b : 0u;
                    m2 |= h == 2 ? b : 0u;
                    m3 |= h == 3 ? b : 0u;
                };
                for (uint32_t q = (j0 & ~3u) + 4 * gl; q < j1; q += 4 * G) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(pk + q);
                    mark(v.x);
                    mark(v.y);
                    mark(v.z);
                    mark(v.w);
                }
            }
        }
        for (uint32_t off = G >> 1; off; off >>= 1) {
            m0 |= __shfl_xor_sync(0xffffffffu, m0, off);
            m1 |= __shfl_xor_sync(0xffffffffu, m1, off);
            m2 |= __shfl_xor_sync(0xffffffffu, m2, off);
            m3 |= __shfl_xor_sync(0xffffffffu, m3, off);
        }
        if (k < ns && gl == 0) done(k, pos, __popc(m0) + __popc(m1) + __popc(m2) + __popc(m3));
    }
}

// A window-edge rank the tile pass could not read off its staged keys.
constexpr uint32_t kRankUnknown = 0xffffffffu;

// Staged keys with time below x (relative to the staged range's start, x
// in [0, span]): the buckets before x's bucket, plus the keys of that bucket
// below x.  The keys of a bucket are contiguous in bucket order and in
// sorted order alike.
template <uint32_t NB, uint32_t SHIFT>
__device__ __forceinline__ uint32_t keys_before(const uint32_t *pk, const uint32_t *cnt, uint32_t n, uint32_t x,
                                                uint32_t bsh, uint32_t span)
{
    if (x >= span) return n;
    const uint32_t b = bucket_of<NB>(x, bsh);
    uint32_t c = cnt[b];
    const uint32_t e = cnt[b + 1];
    for (uint32_t m = c; m < e; ++m) c += (pk[m] >> SHIFT) < x;
    return c;
}

// Level 0 for the key at position i: some window [t_j, t_j + TW) with
// t_i - TW < t_j <= t_i holds at least N hits.  The hits of a window are the
// difference of two exact ranks, so the keys of a bucket need no order; the
// whole buckets inside the window that starts at t_i already hold N hits
// where the tower is busy.  Every hit within TW of a core hit is staged (the
// tile halo covers TW).
template <uint32_t NB, class CTX>
__device__ __noinline__ bool level0_pass(const CTX &cx, uint32_t n, uint32_t i, uint32_t N, uint32_t TW, uint32_t bsh,
                                         uint32_t span)
{
    const uint32_t *pk = cx.pk(), *cnt = cx.cnt();
    const uint32_t ts = CTX::key_t(pk[i]);
    const uint32_t b0 = (ts >> bsh) + 1u, b1 = bucket_of<NB>(ts + TW, bsh);
    if (b1 > b0 && cnt[b1] - cnt[b0] >= N) return true;
    auto busy = [&](uint32_t tj) {
        return keys_before<NB, CTX::kShift>(pk, cnt, n, tj + TW, bsh, span) -
                   keys_before<NB, CTX::kShift>(pk, cnt, n, tj, bsh, span) >=
               N;
    };
    if (busy(ts)) return true;
    // the windows that start at an earlier hit; those of a bucket are looked at
    // one by one only if all the buckets they may touch hold N hits together
    // (else hits that share a few buckets, as under a coarse clock, would each
    // be counted against all of them)
    const uint32_t lo = ts >= TW ? ts - TW + 1u : 0u;
    for (uint32_t b = lo >> bsh; b < b0; ++b) {
        const uint32_t j0 = cnt[b], j1 = cnt[b + 1];
        if (j0 == j1 || cnt[bucket_of<NB>(((b + 1u) << bsh) - 1u + TW, bsh) + 1u] - j0 < N) continue;
        for (uint32_t j = j0; j < j1; ++j) {
            const uint32_t tj = CTX::key_t(pk[j]);
            if (tj >= lo && tj < ts && busy(tj)) return true;
        }
    }
    return false;
}

// The same with hits of at least N different PMTs (up to 128 PMTs; above,
// level0_distinct_warp), on sorted keys: the window slides back start by
// start, keeping per-PMT counts, so it reads each hit within 2 TW once.
template <class CTX>
__device__ __noinline__ bool level0_distinct(const uint32_t *pk, uint32_t n, uint32_t i, uint32_t N, uint32_t TW)
{
    const uint32_t ts = CTX::key_t(pk[i]);
    uint32_t j = i;
    while (j > 0 && CTX::key_t(pk[j - 1]) == ts) --j;             // first index of t_i
    uint16_t cnt[128];
    for (uint32_t p = 0; p < 128; ++p) cnt[p] = 0;
    uint32_t distinct_n = 0, e = j;
    for (;;) {
        const uint32_t tj = CTX::key_t(pk[j]);
        while (e < n && CTX::key_t(pk[e]) - tj < TW) {                // extend the end
            if (cnt[CTX::key_p(pk[e]) & 127u]++ == 0) ++distinct_n;
            ++e;
        }
        if (distinct_n >= N) return true;
        if (j == 0) return false;
        const uint32_t tp = CTX::key_t(pk[j - 1]);
        if (ts - tp >= TW) return false;
        // the previous start: add its hits, drop hits at or past tp + TW
        uint32_t nj = j - 1;
        while (nj > 0 && CTX::key_t(pk[nj - 1]) == tp) --nj;
        for (uint32_t q = nj; q < j; ++q)
            if (cnt[CTX::key_p(pk[q]) & 127u]++ == 0) ++distinct_n;
        while (e > j && CTX::key_t(pk[e - 1]) - tp >= TW) {
            --e;
            if (--cnt[CTX::key_p(pk[e]) & 127u] == 0) --distinct_n;
        }
        j = nj;
    }
}

// Level 0 with distinct PMTs above 128 PMTs, by a warp: the same window
// starts as level0_pass (each first index of a time within TW before t_i),
// each window's PMTs marked in the warp's 4096-bit set in shared memory and
// counted; the first window with N different PMTs ends the search.
template <class CTX>
__device__ __noinline__ bool level0_distinct_warp(const uint32_t *pk, uint32_t n, uint32_t i, uint32_t N, uint32_t TW,
                                                  uint32_t P, uint32_t *set)
{
    const uint32_t lane = lane_id(), nwords = (P + 31u) >> 5;
    const uint32_t ts = CTX::key_t(pk[i]);
    uint32_t j = i;
    while (j > 0 && CTX::key_t(pk[j - 1]) == ts) --j;             // first index of t_i
    for (;;) {
        const uint32_t tj = CTX::key_t(pk[j]);
        for (uint32_t w = lane; w < nwords; w += 32) set[w] = 0u;
        __syncwarp();
        // the window [t_j, t_j + TW): keys from j on, in time order
        for (uint32_t k0 = j; k0 < n; k0 += 32) {
            const uint32_t k = k0 + lane;
            bool in = false;
            if (k < n) {
                const uint32_t kk = pk[k], pj = CTX::key_p(kk);
                in = CTX::key_t(kk) - tj < TW;
                if (in && CHECK(27, pj, P)) atomicOr(&set[pj >> 5], 1u << (pj & 31u));
            }
            if (!__any_sync(0xffffffffu, in)) break;
        }
        __syncwarp();
        uint32_t c = 0;
        for (uint32_t w = lane; w < nwords; w += 32) c += __popc(set[w]);
        c = __reduce_add_sync(0xffffffffu, c);
        __syncwarp();                                       // the set is read before it is cleared again
        if (c >= N) return true;
        if (j == 0) return false;
        const uint32_t tp = CTX::key_t(pk[j - 1]);
        if (ts - tp >= TW) return false;
        for (--j; j > 0 && CTX::key_t(pk[j - 1]) == tp; --j) {
        }
    }
}

// Bucket shift of a staged range of `span` ns: buckets of 2^bsh ns, NBK of
// them cover the range.
template <uint32_t NB>
__device__ __forceinline__ uint32_t bucket_shift(uint32_t span)
{
    const uint32_t top = span > 1 ? 32u - __clz(span - 1u) : 0u;      // bits of span - 1
    const uint32_t nb_bits = 31u - __clz(NB);
    return top > nb_bits ? top - nb_bits : 0u;
}

// Causal count c(s) = #{ j : |t_j - t_s| <= min(dt_max[p_s][p_j], W) } over
// each seed's scan range keys [j0, j1) (seed_range), a group of 2^lg lanes
// per seed; a fired seed sets its position in mask.
//
// Bound by the issue slots and the shared-memory reads of its inner loop (the
// row lookups of 32 lanes meet in 3.4 banks' turns), so a key costs six
// instructions: a quarter of a 16-byte key load, the row
// lookup whose address is one logical operation (kDtRow-aligned rows, the
// key's low byte is the offset in the row), shift, absolute difference,
// compare, count.  No key outside [j0, j1) can pass: those before j0 lie in
// earlier buckets, more than dmax_row(p_s) >= dt before t_s, those from j1
// on in later buckets, and the four end keys past the last key are beyond
// any dt as well, so whole groups of four from j0 rounded down are taken.
template <uint32_t NB, int NC, bool EXT, class C>
__device__ __forceinline__ void count_seeds(const C &cx, uint32_t n, uint32_t ns, uint32_t bsh, uint32_t lg,
                                            uint32_t threshold, uint32_t dt_mask)
{
    const uint32_t tid = threadIdx.x, G = 1u << lg, gl = tid & (G - 1u), gid = tid >> lg, NG = NC >> lg;
    const uint32_t *pk = cx.pk();
    const uint32_t *seeds = cx.seeds();
    const uint32_t rounds = (ns + NG - 1) / NG;
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t k = r * NG + gid;
        uint32_t c = 0, e = 0;
        if (k < ns) {
            e = seeds[k];
            const uint32_t ks = pk[e & 0xffffu];
            const uint32_t ts = C::key_t(ks), ps = C::key_p(ks);
            uint32_t j0, j1;
            seed_range<NB>(cx, ts, ps, bsh, j0, j1);
            if (CHECK(12, j1, n + 1) && CHECK(13, ps, cx.P)) {
                const auto row = cx.row(ps);
                auto causal = [&](uint32_t kj) -> uint32_t {
                    if (!CHECK(11, C::key_p(kj), cx.P)) return 0u;
                    const uint32_t lim = EXT ? row.at(kj) & dt_mask : row.at(kj);
                    return __usad(C::key_t(kj), ts, 0u) <= lim;
                };
                uint32_t ca = 0, cb = 0, cc = 0, cd = 0;
                for (uint32_t q = (j0 & ~3u) + 4 * gl; q < j1; q += 4 * G) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(pk + q);
                    ca += causal(v.x);
                    cb += causal(v.y);
                    cc += causal(v.z);
                    cd += causal(v.w);
                }
                c = ca + cb + cc + cd;
            }
        }
        for (uint32_t off = G >> 1; off; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
        if (k < ns && gl == 0) {
            cx.counts()[k] = (uint16_t)c;
            if (c >= threshold) {
                const uint32_t pos = e & 0xffffu;
                if (!EXT) cx.fired_charge()[pos] = (uint16_t)(e >> 16);
                atomicOr(&cx.mask()[pos >> 5], 1u << (pos & 31u));
            }
        }
    }
}

// One staged tile through the whole trigger: the n records of `stage` (16
// bytes each, any order) span [tb, tb + span); the core is t - tb in
// [lo_t, hi_t).  The default builds take the default seed rule alone; the
// extended ones (EXT) level 0, seed rule 1, the distinct count, row outputs
// and event extraction as well (on 52 M hits with dt rows in shared memory
// and unsorted buckets where order is not needed: the ladder 4.61 ms, 5.38
// with a full sort and dt rows through the cache, the distinct count 1.67,
// 2.30 before, both in 4096-hit tiles).
//
//  A. every record becomes a packed key (TileCtx::key), is counted in its
//     time bucket (t - tb) >> bsh and marked in its floor cell (floor, and
//     time in steps of 2^csh > tau: two bits, one hit and more than one);
//  B. bucket offsets (exclusive scan of the counts), and a mark on each floor
//     cell with another hit in it or in a neighbouring cell;
//  C. the k-way merge of the PMT runs ("DAQ system of NEMO Phase II"): keys
//     scattered to bucket order, about one key per bucket.  A core hit
//     over the charge threshold or in a marked cell becomes a candidate.
//     For row outputs and level 0 over different PMTs the keys of a bucket
//     are also sorted by (t, pmt, charge);
//  D. floor coincidences ("Sorting and triggering in GPU": another PMT of
//     the same floor within tau): each candidate looks through the buckets
//     of [t - tau, t + tau].  EXT: or for seed rule 1 (coincidence_seed; it
//     needs a hit of its own floor within SC or FC), and level 0 tests each
//     seed;
//  E. the causal counts (count_seeds);
//  F. the fired seeds to out, in (t, pmt, charge) order: a seed's rank is
//     the number of fired positions before it, corrected inside its bucket.
//
// Bound by the shared-memory pipe (65 % busy) and the latency of the phases'
// chains of lookups, then by instruction issue (59 %), not by HBM (13 %).  So
// each phase reads shared memory as seldom as it can: the floor cells leave
// about one hit in six for phase D's search (a search from every hit took a
// third of the pass), charges travel with the candidates instead of being
// scattered with every key, and two lanes share a seed's emission.  The 64
// slices of both towers (205 M hits, tiles of 2048 at 90 and 95 %) take 3.61
// ms, 4.43 ms with the search from every hit and an ordered seed list; the
// 2688-PMT slice 0.96 ms (4096 at 90 %; 1.12 in tiles of 2048), 2.05 before.
// The bucket counts, cells and mask are zero on entry and on return.
template <int CAP, int NC, bool NARROW, bool EXT, bool DENSE, bool CROWD = false>
__device__ CoreOut tile_pass(TileCtx<CAP, NC, NARROW, EXT, CROWD> &cx, const uint64_t *stage, uint32_t n, int64_t tb,
                             uint32_t span, uint32_t lo_t, uint32_t hi_t, const TrigParams &tp, trig_trigger *out,
                             uint32_t *wr, bool out_at_c0, uint32_t rank_base, int64_t dbg_rank_lo, uint64_t *release_bar)
{
    using C = TileCtx<CAP, NC, NARROW, EXT, CROWD>;
    using L = typename C::L;
    constexpr uint32_t NW = NC / 32;
    constexpr int PER = CAP / NC;
    constexpr uint32_t NB = L::NBK;
    constexpr uint32_t M = L::kCells;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5, lt = (1u << lane) - 1u;
    const uint32_t bsh = bucket_shift<NB>(span);
    const uint32_t tau = tp.tau;
    __shared__ uint32_t s_red[NW];
    __shared__ uint32_t s_n[4];             // candidates, seeds, keys before the core, before its end
    uint32_t *cnt = cx.cnt(), *mask = cx.mask(), *cells = cx.cells();
    uint32_t *pk = cx.pk(), *seeds = cx.seeds(), *cand = cx.cand();
    const uint16_t *fl = cx.floor_s();
    // floor cells of 2^csh ns, more than the floor coincidence (under seed
    // rule 1, the wider of SC and FC); the floors' ranges of cells follow
    // each other, taken modulo M (two hits that share a cell by chance only
    // cost a search)
    const bool rule1 = EXT && tp.seed_rule == 1;
    const uint32_t csh = 32u - __clz(rule1 ? max(tp.sc_w, tp.fc_w) : tau), fstep = (span >> csh) + 2u;
#ifdef TRIG_PHASE_STATS
    long long t_ph = clock64();
#define PHASE_MARK(i)                                   \
    do {                                                \
        if (tid == 0) {                                 \
            const long long now_ = clock64();           \
            PHASE_ADD((i), now_ - t_ph);                \
            t_ph = now_;                                \
        }                                               \
    } while (0)
#else
#define PHASE_MARK(i) ((void)0)
#endif

    // level 0 over different PMTs and the row outputs need the keys of a
    // bucket in order
    const bool sorted = EXT && ((tp.l0_hits && tp.l0_distinct) || tp.dbg_merged);

    // A. keys, bucket counts, floor cells
    uint32_t key[PER], cs[PER], hc[PER];  // packed key; charge << 16 | slot in the bucket; floor cell
    if (tid == 0) s_n[0] = s_n[1] = 0;
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        const uint32_t i = tid + r * NC;
        key[r] = kPkNone;
        cs[r] = hc[r] = 0;
        if (i < n) {
            uint32_t tr, pq;            // time from tb, PMT and charge
            if (CROWD) {
                const uint2 v = *reinterpret_cast<const uint2 *>(stage + i);
                tr = v.x, pq = v.y;
            } else {
                const uint4 v = *reinterpret_cast<const uint4 *>(stage + 2 * i);
                // in 32 bits (the staged range spans less than 2^20 ns)
                tr = min(v.x - (uint32_t)tb, span - 1u), pq = v.z;
            }
            const uint32_t p = pq & 0xfffu;
            key[r] = C::key(tr, p);
            cs[r] = (pq & 0xffff0000u) | atomicAdd(&cnt[tr >> bsh], 1u);
            const uint32_t h = (fl[p] * fstep + (tr >> csh)) & (M - 1u), bit = 1u << (2u * (h & 15u));
            hc[r] = h;
            if (atomicOr(&cells[h >> 4], bit) & bit) atomicOr(&cells[h >> 4], bit << 1);
        }
    }
    // the stage buffer has been read: order those reads before the
    // producer's next bulk copy into it, then hand it back
    if (release_bar) fence_proxy_async_smem();
    cons_sync<NC>();
    if (release_bar && tid == 0) mbar_arrive(release_bar);
    PHASE_MARK(kPhA);

    // B. bucket offsets; and each floor cell's two bits become one: another
    //    hit in the cell, or one in a neighbouring cell
    {
        constexpr uint32_t MV = M / 64 / NC;              // 16-byte vectors of cells per thread
        static_assert(M % (64 * NC) == 0, "each thread folds whole 16-byte vectors of cells");
        uint4 *m4 = reinterpret_cast<uint4 *>(cells) + tid * MV;
        uint32_t fold[4 * MV];
        {
            uint32_t prev = cells[(tid * 4 * MV - 1u) & (M / 16 - 1u)];
            const uint32_t last = cells[(tid * 4 * MV + 4 * MV) & (M / 16 - 1u)];
            uint32_t w[4 * MV + 1];
#pragma unroll
            for (uint32_t i = 0; i < MV; ++i) {
                const uint4 c = m4[i];
                w[4 * i] = c.x, w[4 * i + 1] = c.y, w[4 * i + 2] = c.z, w[4 * i + 3] = c.w;
            }
            w[4 * MV] = last;
#pragma unroll
            for (uint32_t i = 0; i < 4 * MV; ++i) {
                fold[i] = (w[i] >> 1) | __funnelshift_l(prev, w[i], 2) | __funnelshift_r(w[i], w[i + 1], 2);
                prev = w[i];
            }
        }
        constexpr uint32_t V = NB / NC / 4;
        static_assert(NB % (4 * NC) == 0, "each thread scans whole 16-byte vectors");
        uint4 *c4 = reinterpret_cast<uint4 *>(cnt) + tid * V;
        uint4 v[V];
        uint32_t local = 0;
#pragma unroll
        for (uint32_t i = 0; i < V; ++i) {
            v[i] = c4[i];
            local += v[i].x + v[i].y + v[i].z + v[i].w;
        }
        const uint32_t incl = warp_incl_scan(local);
        if (lane == 31) s_red[warp] = incl;
        cons_sync<NC>();
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? s_red[lane % NW] : 0u);
        uint32_t run = before + incl - local;
#pragma unroll
        for (uint32_t i = 0; i < V; ++i) {
            uint4 o;
            o.x = run;
            o.y = o.x + v[i].x;
            o.z = o.y + v[i].y;
            o.w = o.z + v[i].z;
            run = o.w + v[i].w;
            c4[i] = o;
        }
#pragma unroll
        for (uint32_t i = 0; i < MV; ++i)
            m4[i] = make_uint4(fold[4 * i], fold[4 * i + 1], fold[4 * i + 2], fold[4 * i + 3]);
        if (tid == NC - 1) cnt[NB] = run;
        if (tid < 4) pk[n + tid] = ~C::kPmtMask;          // end keys (the last time, PMT 0)
    }
    cons_sync<NC>();
    PHASE_MARK(kPhB);

    // C. bucket order and candidates (charge << 16 | position, with bit 15
    //    set for a charge over the threshold); where they are needed sorted,
    //    each key then goes to its rank inside its bucket, in place
    {
        uint32_t pos[PER];
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            pos[r] = 0;
            if (key[r] != kPkNone) {
                pos[r] = cnt[C::key_t(key[r]) >> bsh] + (cs[r] & 0xffffu);
                if (CHECK(22, pos[r], CAP)) {
                    pk[pos[r]] = key[r];
                    if (EXT) cx.chg()[pos[r]] = (uint16_t)(cs[r] >> 16);
                }
            }
        }
        if (sorted) {
            const uint16_t *chg = cx.chg();
            cons_sync<NC>();
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                if (key[r] == kPkNone) continue;
                const uint32_t k = key[r], b = C::key_t(k) >> bsh, q = cs[r] >> 16;
                const uint32_t s0 = cnt[b], s1 = cnt[b + 1];
                uint32_t rk = s0;
                if (s1 - s0 > 1)
                    for (uint32_t m = s0; m < s1; ++m) {
                        const uint32_t o = pk[m];
                        rk += o < k;
                        if (o == k && m != pos[r]) rk += chg[m] < q || (chg[m] == q && m < pos[r]);   // equal time, PMT
                    }
                pos[r] = rk;
            }
            cons_sync<NC>();
#pragma unroll
            for (int r = 0; r < PER; ++r)
                if (key[r] != kPkNone && CHECK(23, pos[r], CAP)) {
                    pk[pos[r]] = key[r];
                    cx.chg()[pos[r]] = (uint16_t)(cs[r] >> 16);
                }
        }
        uint32_t m[PER], total = 0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            bool c = false;
            if (key[r] != kPkNone) {
                const uint32_t tr = C::key_t(key[r]);
                if (tr - lo_t < hi_t - lo_t) {
                    const bool over = !rule1 && (cs[r] >> 16) >= tp.q_seed;
                    c = over || ((cells[hc[r] >> 4] >> (2u * (hc[r] & 15u))) & 1u);
                    cs[r] = (cs[r] & 0xffff0000u) | pos[r] | (over ? 0x8000u : 0u);
                }
            }
            m[r] = __ballot_sync(0xffffffffu, c);
            total += __popc(m[r]);
        }
        uint32_t at = 0;
        if (lane == 0 && total) at = atomicAdd(&s_n[0], total);
        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            if ((m[r] >> lane) & 1u) cand[at + __popc(m[r] & lt)] = cs[r];
            at += __popc(m[r]);
        }
    }
    cons_sync<NC>();
    PHASE_MARK(kPhC);

    // D. floor coincidences of the candidates, four keys of the range at a
    //    time; the seeds take the cells' place
    {
        const uint32_t nc = s_n[0];
        for (uint32_t x = warp * 32; x < nc; x += NC) {
            bool seed = false;
            uint32_t e = 0;
            if (x + lane < nc) {
                e = cand[x + lane];
                seed = (e >> 15) & 1u;
                e &= 0xffff7fffu;
                if (rule1) seed = coincidence_seed<NB>(cx, tp, e & 0xffffu, bsh);
                else if (!seed) {
                    const uint32_t ki = pk[e & 0xffffu], ti = C::key_t(ki), pi = C::key_p(ki), fi = fl[pi];
                    uint32_t j = cnt[(ti > tau ? ti - tau : 0u) >> bsh];
                    const uint32_t je = cnt[bucket_of<NB>(ti + tau, bsh) + 1];
                    for (; j < je; j += 4) {
                        uint32_t kj[4], fj[4];
#pragma unroll
                        for (uint32_t u = 0; u < 4; ++u) kj[u] = pk[min(j + u, je - 1u)];
#pragma unroll
                        for (uint32_t u = 0; u < 4; ++u) fj[u] = fl[C::key_p(kj[u])];
#pragma unroll
                        for (uint32_t u = 0; u < 4; ++u)
                            seed = seed || (__usad(C::key_t(kj[u]), ti, 0u) <= tau && C::key_p(kj[u]) != pi && fj[u] == fi);
                    }
                }
            }
            if (EXT && tp.l0_hits) {
                // level 0 (N hits within TW) before the seed triggers count
                if (tp.l0_distinct && cx.P > 128) {
                    // a warp per seed, marking its PMTs in a shared-memory set
                    for (uint32_t todo = __ballot_sync(0xffffffffu, seed); todo; todo &= todo - 1u) {
                        const uint32_t b = __ffs(todo) - 1;
                        const uint32_t i = __shfl_sync(0xffffffffu, e, b) & 0xffffu;
                        const bool ok = level0_distinct_warp<C>(pk, n, i, tp.l0_hits, tp.l0_window, cx.P, cx.pmt_set(warp));
                        if (lane == b) seed = ok;
                    }
                } else if (seed) {
                    seed = tp.l0_distinct ? level0_distinct<C>(pk, n, e & 0xffffu, tp.l0_hits, tp.l0_window)
                                          : level0_pass<NB>(cx, n, e & 0xffffu, tp.l0_hits, tp.l0_window, bsh, span);
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, seed);
            uint32_t at = 0;
            if (lane == 0 && m) at = atomicAdd(&s_n[1], __popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (seed && CHECK(2, at + __popc(m & lt), CAP)) seeds[at + __popc(m & lt)] = e;
        }
        // keys before the core: the fired seeds' place in the slice's staging
        if (tid == NC - 1) s_n[2] = keys_before<NB, C::kShift>(pk, cnt, n, lo_t, bsh, span);
        if (EXT && tid == NC - 33) s_n[3] = keys_before<NB, C::kShift>(pk, cnt, n, hi_t, bsh, span);
    }
    cons_sync<NC>();
    PHASE_MARK(kPhD);
    const uint32_t ns = s_n[1], c0 = s_n[2];
    if (tid == 0) PHASE_ADD(kPhSeeds, ns);

    // E. causal counts: the dense builds (hundreds of keys per seed) take a
    //    warp per seed; the others four lanes, or more while all seeds of
    //    the tile still fit in one round
    uint32_t lg = 5;
    if (!DENSE) {
        lg = 2;
        while (lg < 5 && (ns << (lg + 1)) <= NC) ++lg;
    }
    if (EXT && tp.count_distinct) count_distinct_pmts<NB, NC>(cx, n, ns, bsh, tp.threshold, tp.dt_mask);
    else count_seeds<NB, NC, EXT>(cx, n, ns, bsh, lg, tp.threshold, tp.dt_mask);
    cons_sync<NC>();
    PHASE_MARK(kPhE);

    // F. each warp counts the fired positions before each mask word (a lane
    //    takes PW consecutive words), then takes 16 seeds at a time, two
    //    lanes per seed: one finds the merged rank of the first hit of the
    //    seed's event window [t - h, t + h], the other of the first hit past
    //    it, where that bound lies in the staged range (else kRankUnknown:
    //    the window pass searches for it)
    constexpr uint32_t PW = CAP / 32 / 32;
    uint32_t wn[PW], own = 0;
#pragma unroll
    for (uint32_t w = 0; w < PW; ++w) {
        wn[w] = __popc(mask[lane * PW + w]);
        own += wn[w];
    }
    const uint32_t incl = warp_incl_scan(own), wpre = incl - own;
    const uint32_t n_fired = __shfl_sync(0xffffffffu, incl, 31);
    const size_t out_at = out_at_c0 ? c0 : 0u;
    for (uint32_t k0 = warp * 16; k0 < ns; k0 += NW * 16) {
        const uint32_t k = k0 + (lane >> 1), side = lane & 1u;
        const uint32_t e = k < ns ? seeds[k] : 0u, c = k < ns ? cx.counts()[k] : 0u;
        const uint32_t pos = e & 0xffffu, w = pos >> 5;
        // fired positions before pos: the words before its word ...
        uint32_t o = __shfl_sync(0xffffffffu, wpre, w / PW);
#pragma unroll
        for (uint32_t x = 0; x + 1 < PW; ++x) {
            const uint32_t v = __shfl_sync(0xffffffffu, wn[x], w / PW);
            o += x < w % PW ? v : 0u;
        }
        if (k >= ns || c < tp.threshold) continue;
        // ... and those before it in the word
        o += __popc(mask[w] & ((1u << (pos & 31u)) - 1u));
        const uint32_t ks = pk[pos], ts = C::key_t(ks), b = ts >> bsh;
        // fired seeds of its bucket that order the other way round
        for (uint32_t j = cnt[b], je = cnt[b + 1]; j < je; ++j) {
            if (j == pos || !((mask[j >> 5] >> (j & 31u)) & 1u)) continue;
            const uint32_t kj = pk[j];
            bool less = kj < ks, more = kj > ks;
            if (kj == ks) {                      // the same time and PMT: by charge
                const uint32_t qj = cx.fired_charge()[j];
                less = qj < (e >> 16);
                more = qj > (e >> 16);
            }
            o += j > pos && less ? 1u : 0u;
            o -= j < pos && more ? 1u : 0u;
        }
        if (!CHECK(3, o, n_fired)) continue;
        const uint32_t wh = tp.win_half, x = side ? ts + wh + 1u : ts - wh;
        const bool known = side ? x <= span : ts >= wh;
        wr[2 * (out_at + o) + side] = known ? rank_base + keys_before<NB, C::kShift>(pk, cnt, n, x, bsh, span) : kRankUnknown;
        // the trigger's two halves: time; PMT, charge and count
        const uint64_t half = side ? (uint64_t)c << 32 | (e & 0xffff0000u) | C::key_p(ks) : (uint64_t)(tb + (int64_t)ts);
        reinterpret_cast<uint64_t *>(out + out_at + o)[side] = half;
    }
    // optional row outputs: the merged core rows (verification, and the
    // merged stream of event extraction) and each row's causal count
    // (verification only); rows are indexed by merged rank minus the rank of
    // the slice's first owned hit
    if (EXT && tp.dbg_merged) {
        const uint32_t c1 = s_n[3];
        const uint64_t dbg_base = (uint64_t)(dbg_rank_lo + (int64_t)c0);
        for (uint32_t i = tid; i < c1 - c0; i += NC) {
            const uint32_t k = pk[c0 + i];
            // (8-byte stores: the rows may be the caller's buffer)
            uint64_t *row = reinterpret_cast<uint64_t *>(tp.dbg_merged + dbg_base + i);
            row[0] = (uint64_t)(tb + (int64_t)C::key_t(k));
            row[1] = C::key_p(k) | (uint32_t)cx.chg()[c0 + i] << 16;
            if (tp.dbg_seedcnt) tp.dbg_seedcnt[dbg_base + i] = 0xffffffffu;
        }
        if (tp.dbg_seedcnt) {
            cons_sync<NC>();
            for (uint32_t k = tid; k < ns; k += NC)
                tp.dbg_seedcnt[dbg_base + ((seeds[k] & 0xffffu) - c0)] = cx.counts()[k];
        }
    }
    // leave the bucket counts, cells and mask zero for the next tile
    cons_sync<NC>();
    PHASE_MARK(kPhF);
    {
        uint4 *z = reinterpret_cast<uint4 *>(cnt);
        uint4 *y = reinterpret_cast<uint4 *>(cells);
        static_assert(M / 16 == NB, "as many words of cells as of bucket counts");
        for (uint32_t i = tid; i < NB / 4; i += NC) z[i] = y[i] = make_uint4(0, 0, 0, 0);
        for (uint32_t i = tid; i < (uint32_t)CAP / 32; i += NC) mask[i] = 0;
    }
    cons_sync<NC>();
    PHASE_MARK(kPhG);
#undef PHASE_MARK
    CoreOut co;
    co.n_fired = n_fired;
    co.n_seeds = ns;
    co.c0 = c0;
    return co;
}

// What a block's shared memory holds for crowd_pass: the library's own tiles
// of 2048 hits take pieces of up to 4096 (the shape untuned detectors always
// had room for); other shapes have none.
template <int CAP, int NC>
constexpr uint32_t kCrowdCap = CAP == 2048 && NC == 512 ? 2u * CAP : CAP;

// A piece of core_ns with n > cap hits is left to crowd_pass if it fits there
// and halving it would not help much: nearly all of its hits are halo.
__device__ __forceinline__ bool crowded(uint64_t n, uint32_t core_ns, uint32_t H, uint32_t crowd_cap)
{
    return n <= crowd_cap && (core_ns == 1 || core_ns <= H / 4u);
}

// A piece [lo, hi) of a core whose hits, halos included, do not fit in a tile
// and whose core cannot usefully be split further: a burst so dense that the
// halos alone nearly fill a tile.  The tile pass on a layout for twice the
// hits, over the whole of the block's memory (the stager's buffer too: the
// stager is done).  The hits of [lo - H, hi + H), at most
// 2 CAP, are collected with plain loads after per-PMT searches.
// 18 k hits of 84 PMTs in 30 us take 2.9 ms, 3.9 in 4096-hit tiles; 2048-hit
// tiles without it refused them.
// Its fired seeds go to the merged rank `at` of the slice's staging (at_c0: to
// that of the first core hit, `at` being the first collected hit's).
template <int CAP, int NC, bool NARROW, bool EXT, bool DENSE>
__device__ CoreOut crowd_pass(const TileCtx<CAP, NC, NARROW, EXT> &host, const SliceDesc &d, int64_t lo, int64_t hi,
                              const TrigParams &tp, uint32_t at, bool at_c0, uint32_t rank_lo)
{
    using C = TileCtx<2 * CAP, NC, NARROW, EXT, true>;
    using L = typename C::L;
    using H = TileLayout<CAP, NC, NARROW, EXT>;
    constexpr uint32_t NW = NC / 32, kCap = 2 * CAP;
    __shared__ uint32_t s_n;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5, P = d.n_pmt;
    C cx;
    cx.P = host.P;
    cx.tab = host.tab;
    cx.pp = host.pp;
    cx.dt_g = host.dt_g;
    auto clear = [&](size_t from, size_t to) {
        uint32_t *w = reinterpret_cast<uint32_t *>(g_tile_smem);
        for (uint32_t i = (uint32_t)from / 4 + tid; i < (uint32_t)to / 4; i += NC) w[i] = 0;
    };
    const int64_t tb = lo - (int64_t)tp.H, te = hi + (int64_t)tp.H;
    if (tid == 0) s_n = 0;
    clear(L::oCell, L::oChg);
    cons_sync<NC>();
    uint2 *rec = reinterpret_cast<uint2 *>(cx.stage());
    for (uint32_t p0 = warp * 32; p0 < P; p0 += NW * 32) {
        uint64_t a = 0;
        uint32_t len = 0;
        if (p0 + lane < P) {
            const uint64_t ep = d.pmt_off[p0 + lane + 1];
            a = lb_time(d.hits, d.pmt_off[p0 + lane], ep, tb);
            len = (uint32_t)(lb_time(d.hits, a, ep, te) - a);
        }
        const uint32_t incl = warp_incl_scan(len);
        uint32_t to = 0;
        if (lane == 31) to = atomicAdd(&s_n, incl);
        to = __shfl_sync(0xffffffffu, to, 31) + incl - len;
        for (uint32_t q = 0; q < 32; ++q) {
            const uint64_t qa = __shfl_sync(0xffffffffu, a, q);
            const uint32_t ql = __shfl_sync(0xffffffffu, len, q), qd = __shfl_sync(0xffffffffu, to, q);
            for (uint32_t e = lane; e < ql; e += 32) {
                const trig_hit h = load_hit(d.hits + qa + e);
                if (qd + e < kCap) rec[qd + e] = make_uint2((uint32_t)(h.t_ns - tb), h.pmt | (uint32_t)h.charge << 16);
            }
        }
    }
    cons_sync<NC>();
    const CoreOut co = tile_pass<kCap, NC, NARROW, EXT, DENSE, true>(
        cx, cx.stage(), min(s_n, kCap), tb, (uint32_t)(te - tb), tp.H, tp.H + (uint32_t)(hi - lo), tp, d.stage + at,
        d.wrank + 2 * (size_t)at, at_c0, rank_lo, (int64_t)rank_lo - (int64_t)d.dbg_rank0, nullptr);
    clear(H::oPk, H::oChg);             // the tile pass's counts, cells and mask
    cons_sync<NC>();
    return co;
}

// Last resort of the tiles that the stager cannot split: a single bucket of a
// wide slice with its halo holds more than CAP hits, or a piece of a narrow
// one is crowded.  Split its core in halves until each piece fits; pieces are
// staged with plain loads after per-PMT binary searches.  A 1 ns core that
// still does not fit, nor in crowd_pass, is reported (TRIG_FLAG_TILE_FULL) and
// skipped.
template <int CAP, int NC, class PASS, class CROWD>
__device__ void tile_overflow(PASS pass, CROWD crowd, uint64_t *buf, const SliceDesc &d, uint32_t g, uint32_t *red, int64_t *stk)
{
    constexpr uint32_t NW = NC / 32;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const uint32_t P = d.n_pmt, H = d.halo;
    const int64_t W = d.tile_w;
    const int64_t Bg = d.t0 + (int64_t)g * W;
    const int64_t core_end = min(Bg + W, d.t0 + d.slice_ns);
    uint64_t *part = reinterpret_cast<uint64_t *>(red + 8);          // [NW]
    uint64_t *part2 = reinterpret_cast<uint64_t *>(red + 8 + 2 * NW);  // [NW]
    // merged rank of the tile's first core hit
    uint64_t rk = 0;
    for (uint32_t p = tid; p < P; p += NC) {
        uint64_t sp = d.pmt_off[p], ep = d.pmt_off[p + 1];
        rk += lb_time(d.hits, sp, ep, Bg) - sp;
    }
    rk = warp_sum_u64(rk);
    if (lane == 0) part[warp] = rk;
    cons_sync<NC>();
    if (tid == 0) {
        uint64_t tot = 0;
        for (uint32_t w = 0; w < NW; ++w) tot += part[w];
        red[4] = (uint32_t)tot;     // tile rank
        red[5] = 0;                 // fired so far
        red[6] = 0;                 // seeds so far
        stk[0] = Bg;
        stk[1] = core_end;
        red[7] = 1;                 // stack depth
    }
    cons_sync<NC>();
    const uint32_t tile_rank = red[4];
    for (int guard = 0; guard < 1 << 20; ++guard) {
        uint32_t depth = red[7];
        if (depth == 0) break;
        const int64_t lo = stk[2 * (depth - 1)], hi = stk[2 * (depth - 1) + 1];
        cons_sync<NC>();
        // extended count and rank of the piece
        uint64_t tot = 0, rlo = 0;
        for (uint32_t p = tid; p < P; p += NC) {
            uint64_t sp = d.pmt_off[p], ep = d.pmt_off[p + 1];
            uint64_t a = lb_time(d.hits, sp, ep, lo - (int64_t)H);
            uint64_t b = lb_time(d.hits, a, ep, hi + (int64_t)H);
            tot += b - a;
            rlo += a - sp;
        }
        tot = warp_sum_u64(tot);
        rlo = warp_sum_u64(rlo);
        if (lane == 0) {
            part[warp] = tot;
            part2[warp] = rlo;
        }
        cons_sync<NC>();
        if (tid == 0) {
            uint64_t T = 0, R = 0;
            for (uint32_t w = 0; w < NW; ++w) {
                T += part[w];
                R += part2[w];
            }
            red[2] = T > 0xffffffffull ? 0xffffffffu : (uint32_t)T;
            red[3] = (uint32_t)R;
            red[7] = depth - 1;                      // pop
            red[1] = T > (uint64_t)CAP && crowded(T, (uint32_t)(hi - lo), H, kCrowdCap<CAP, NC>);
            if (T > (uint64_t)CAP && !red[1]) {
                if (hi - lo > 1 && depth + 1 < 64) {
                    int64_t mid = lo + (hi - lo) / 2;
                    stk[2 * (depth - 1)] = mid;          // right half below ...
                    stk[2 * (depth - 1) + 1] = hi;
                    stk[2 * depth] = lo;                 // ... left half on top
                    stk[2 * depth + 1] = mid;
                    red[7] = depth + 1;
                } else {
                    report(d, TRIG_FLAG_TILE_FULL);
                }
            }
        }
        cons_sync<NC>();
        const uint32_t total = red[2], rank_lo = red[3];
        if (red[1]) {
            const uint32_t fired0 = red[5];
            const CoreOut co = crowd(lo, hi, tile_rank + fired0, false, rank_lo);
            if (tid == 0) {
                red[5] = fired0 + co.n_fired;
                red[6] += co.n_seeds;
            }
            cons_sync<NC>();
            continue;
        }
        if (total > (uint32_t)CAP) continue;         // split (or skipped)
        // stage the piece: PMTs in order, warps take groups of 32 PMTs
        uint32_t dst = 0;
        for (uint32_t p0 = 0; p0 < P; p0 += 32) {
            uint32_t p = p0 + lane;
            uint64_t a = 0, len = 0;
            if (p < P) {
                uint64_t sp = d.pmt_off[p], ep = d.pmt_off[p + 1];
                a = lb_time(d.hits, sp, ep, lo - (int64_t)H);
                len = lb_time(d.hits, a, ep, hi + (int64_t)H) - a;
            }
            uint32_t incl = warp_incl_scan((uint32_t)len);
            uint32_t my = dst + incl - (uint32_t)len;
            if (((p0 >> 5) % NW) == warp) {
                for (uint32_t q = 0; q < 32; ++q) {
                    uint64_t qa = __shfl_sync(0xffffffffu, a, q);
                    uint32_t ql = __shfl_sync(0xffffffffu, (uint32_t)len, q);
                    uint32_t qd = __shfl_sync(0xffffffffu, my, q);
                    for (uint32_t e = lane; e < ql; e += 32) {
                        trig_hit h = load_hit(d.hits + qa + e);
                        if (!CHECK(4, qd + e, CAP) || !CHECK(5, qa + e, d.n_hits)) continue;
                        buf[2 * (qd + e)] = (uint64_t)h.t_ns;
                        buf[2 * (qd + e) + 1] = (uint64_t)h.pmt | ((uint64_t)h.charge << 16);
                    }
                }
            }
            dst += __shfl_sync(0xffffffffu, incl, 31);
        }
        cons_sync<NC>();
        const int64_t tb = lo - (int64_t)H;
        const uint32_t span = (uint32_t)(hi - lo) + 2 * H;
        const uint32_t fired0 = red[5];
        CoreOut co = pass(buf, total, tb, span, H, H + (uint32_t)(hi - lo), d.stage + tile_rank + fired0,
                          d.wrank + 2 * (size_t)(tile_rank + fired0), false, rank_lo,
                          (int64_t)rank_lo - (int64_t)d.dbg_rank0);
        if (tid == 0) {
            red[5] = fired0 + co.n_fired;
            red[6] += co.n_seeds;
        }
        cons_sync<NC>();
    }
    if (tid == 0) {
        d.tile_nfired[g] = red[5];
        d.tile_rank[g] = tile_rank;
        atomicAdd(reinterpret_cast<unsigned long long *>(&d.stats->n_seeds), (unsigned long long)red[6]);
    }
    cons_sync<NC>();
}

// A tile put off (k_tile).  Where its code stands decides how many of the tile
// pass's registers it costs in builds of 56 a thread: in the extended ones it
// is inlined after the loop over the tiles, with crowd_pass a call (16 slices
// with events 2.01 ms, 2.05 all inlined, 2.08 all a call, 1.99 without any of
// it), in the default ones one call (a 320 k-hit slice 31.4, 32.4, 31.4, 31.6 us;
// 64 slices 4.79, 4.76, 4.79, 4.73 ms).
template <int CAP, int NC, bool NARROW, bool EXT, bool DENSE>
__device__ __noinline__ void crowd_call(uint32_t pmts, uint32_t tab, uint32_t pp, const uint16_t *dt_g, const SliceDesc *d, int64_t lo,
                                        int64_t hi, const TrigParams *tp, uint32_t at, bool at_c0, uint32_t rank_lo, CoreOut *res)
{
    TileCtx<CAP, NC, NARROW, EXT> cx;
    cx.P = pmts, cx.tab = tab, cx.pp = pp, cx.dt_g = dt_g;
    const CoreOut co = crowd_pass<CAP, NC, NARROW, EXT, DENSE>(cx, *d, lo, hi, *tp, at, at_c0, rank_lo);
    if (threadIdx.x == 0) *res = co;
    cons_sync<NC>();
}

template <int CAP, int NC, bool NARROW, bool EXT, bool DENSE>
__device__ __forceinline__ void put_off_tile(TileCtx<CAP, NC, NARROW, EXT> &cx, const SliceDesc &d, uint32_t g, const TrigParams &tp)
{
    __shared__ __align__(16) uint32_t red[64 + 64];
    __shared__ int64_t stk[128];
    __shared__ CoreOut res;
    auto pass = [&](const uint64_t *stage, uint32_t n, int64_t tb, uint32_t span, uint32_t lo_t, uint32_t hi_t, trig_trigger *out,
                    uint32_t *wr, bool out_at_c0, uint32_t rank_base, int64_t dbg_rank_lo) {
        return tile_pass<CAP, NC, NARROW, EXT, DENSE>(cx, stage, n, tb, span, lo_t, hi_t, tp, out, wr, out_at_c0, rank_base,
                                                      dbg_rank_lo, nullptr);
    };
    auto crowd = [&](int64_t lo, int64_t hi, uint32_t at, bool at_c0, uint32_t rank_lo) {
        if constexpr (kCrowdCap<CAP, NC> == CAP) return CoreOut{};
        else if constexpr (EXT) {
            crowd_call<CAP, NC, NARROW, EXT, DENSE>(cx.P, cx.tab, cx.pp, cx.dt_g, &d, lo, hi, &tp, at, at_c0, rank_lo, &res);
            return res;
        } else return crowd_pass<CAP, NC, NARROW, EXT, DENSE>(cx, d, lo, hi, tp, at, at_c0, rank_lo);
    };
    tile_overflow<CAP, NC>(pass, crowd, cx.stage(), d, g, red, stk);
}

template <int CAP, int NC, bool NARROW, bool EXT, bool DENSE>
__device__ __noinline__ void put_off_call(uint32_t pmts, uint32_t tab, uint32_t pp, const uint16_t *dt_g, const SliceDesc *d, uint32_t g,
                                          const TrigParams *tp)
{
    TileCtx<CAP, NC, NARROW, EXT> cx;
    cx.P = pmts, cx.tab = tab, cx.pp = pp, cx.dt_g = dt_g;
    put_off_tile<CAP, NC, NARROW, EXT, DENSE>(cx, *d, g, *tp);
}

// The stager's side of the hand-over of the one staging buffer.
struct Stager {
    uint64_t *full, *empty;
    ItemInfo *info;
    uint64_t *stage;
    uint32_t it;                // hand-overs so far
    // lane 0 waits (bounded) for the buffer and decides for the warp
    __device__ __forceinline__ bool wait_free(BatchHeader *hdr, uint64_t wait_ns)
    {
        uint32_t ok = 1;
        if (it >= 1 && lane_id() == 0) {
#ifdef TRIG_PHASE_STATS
            const long long tw0 = clock64();
            uint32_t pr = 0;
            ok = mbar_wait(empty, (it - 1) & 1u, wait_ns, &pr) ? 1u : 0u;
            PHASE_ADD(kPhProdWait, clock64() - tw0);
            PHASE_ADD(kPhProdWaitRounds, pr);
#else
            ok = mbar_wait(empty, (it - 1) & 1u, wait_ns) ? 1u : 0u;
#endif
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
        if (!ok && lane_id() == 0) atomicOr(&hdr->err, TRIG_FLAG_TIMEOUT);
        ++it;
        return ok != 0;
    }
    // the item's description; with n > 0 hits to come by bulk copies
    __device__ __forceinline__ void hand_over(const ItemInfo &x, uint32_t n)
    {
        if (lane_id() == 0) {
            *info = x;
            info->n = n;
            if (n) mbar_arrive_expect_tx(full, n * 16u);
            else mbar_arrive(full);
        }
        __syncwarp();
    }
    // one copy of a PMT run of len hits from a, at dst of the tile's (the
    // lanes' runs follow each other); dst moves past the warp's
    __device__ __forceinline__ void copy_run(const trig_hit *hits, uint64_t n_hits, uint32_t a, uint32_t len, uint32_t cap,
                                             uint32_t &dst)
    {
        const uint32_t incl = warp_incl_scan(len);
        if (len && CHECK(6, dst + incl, cap + 1) && CHECK(7, (uint64_t)a + len, n_hits + 1))
            bulk_g2s(stage + 2 * (size_t)(dst + incl - len), hits + a, len * 16u, full);
        dst += __shfl_sync(0xffffffffu, incl, 31);
    }
};

constexpr uint32_t kStageRuns = 4;          // PMT runs per lane of the stager (narrow slices have at most 128)
constexpr uint32_t kMaxPieces = 24;         // open halves of a core below 2^20 ns

// A tile of a narrow slice with more hits than fit (a burst): its core is
// halved until each piece fits with its halo; the pieces' runs are found
// inside the tile's (runs: start and end of each PMT's, in shared memory).  A
// tile with a crowded piece is put off; a 1 ns piece that fits nowhere is
// reported and left out.  Returns false when a wait ran out.
__device__ __forceinline__ bool stage_pieces(Stager &sg, ItemInfo x, uint32_t cap, uint32_t crowd_cap, const SliceDesc *d,
                                          const uint2 *runs, uint2 *pieces, BatchHeader *hdr)
{
    const uint32_t lane = lane_id(), H = d->halo, rlo = x.rank_lo;
    const uint64_t wait_ns = hdr->wait_ns;
    const int64_t Bg = d->t0 + (int64_t)x.g * d->tile_w;
    uint32_t depth = 1;
    if (lane == 0) pieces[0] = make_uint2(0u, x.core);
    __syncwarp();
    while (depth) {
        const uint32_t lo = pieces[depth - 1].x, hi = pieces[depth - 1].y;
        __syncwarp();
        --depth;
        uint32_t pa[kStageRuns], pe[kStageRuns], n = 0, rank = 0;
#pragma unroll
        for (uint32_t r = 0; r < kStageRuns; ++r) {
            const uint2 run = runs[r * 32 + lane];
            pa[r] = (uint32_t)lb_time(d->hits, run.x, run.y, Bg + lo - (int64_t)H);
            pe[r] = (uint32_t)lb_time(d->hits, pa[r], run.y, Bg + hi + (int64_t)H);
            n += pe[r] - pa[r];
            rank += pa[r] - run.x;
        }
        n = __reduce_add_sync(0xffffffffu, n);
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (n > cap) {
            if (cap < crowd_cap && crowded(n, hi - lo, H, crowd_cap)) {
                if (!sg.wait_free(hdr, wait_ns)) return false;
                x.mode = kItemDefer;
                sg.hand_over(x, 0);
                return true;
            } else if (hi - lo > 1 && depth + 2 <= kMaxPieces) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if (lane == 0) {
                    pieces[depth] = make_uint2(mid, hi);            // right half below,
                    pieces[depth + 1] = make_uint2(lo, mid);        // left half on top
                }
                __syncwarp();
                depth += 2;
            } else if (lane == 0) {
                report(*d, TRIG_FLAG_TILE_FULL);
            }
            continue;
        }
        if (n == 0) continue;
        if (!sg.wait_free(hdr, wait_ns)) return false;
        x.rank_lo = rlo + rank;
        x.off = lo, x.core = hi - lo, x.lo_t = H, x.span = hi - lo + 2 * H;
        sg.hand_over(x, n);
        uint32_t dst = 0;
#pragma unroll
        for (uint32_t r = 0; r < kStageRuns; ++r) sg.copy_run(d->hits, d->n_hits, pa[r], pe[r] - pa[r], cap, dst);
    }
    if (!sg.wait_free(hdr, wait_ns)) return false;
    x.mode = kItemEnd;
    sg.hand_over(x, 0);
    return true;
}

// The staged buckets [b_lo, b_hi) of a wide slice's core buckets [c, c + k).
struct BucketRange {
    uint32_t b_lo, b_hi, lead;
    __device__ __forceinline__ BucketRange(const SliceDesc *d, uint32_t c, uint32_t k)
        : b_lo(c > d->bkt_halo ? c - d->bkt_halo : 0u), b_hi(min(c + k + d->bkt_halo, d->n_bkt)), lead(c - b_lo)
    {
    }
    __device__ __forceinline__ uint32_t hits(const SliceDesc *d) const
    {
        if (!CHECK(28, max(b_lo, b_hi), d->n_bkt + 1u)) return 0;
        return __ldg(d->bkt_off + b_hi) - __ldg(d->bkt_off + b_lo);
    }
};

// Buckets of a tile's core: the slice's last tile may end before its width.
__device__ __forceinline__ uint32_t core_buckets(const SliceDesc *d, uint32_t core)
{
    return (core + d->bkt_w - 1u) / d->bkt_w;
}

// A wide slice's tile with more hits than fit (a muon in a full tile): the
// largest piece of its core buckets, halved from all of them, that fits
// everywhere in the core; 0 if not even one bucket does.
__device__ __forceinline__ uint32_t piece_buckets(const SliceDesc *d, uint32_t c_lo, uint32_t core, uint32_t cap)
{
    const uint32_t m = core_buckets(d, core);
    for (uint32_t k = m;; k = (k + 1) / 2) {
        uint32_t most = 0;
        for (uint32_t j = 0; j < m; j += k) most = max(most, BucketRange(d, c_lo + j, min(k, m - j)).hits(d));
        if (most <= cap) return k;
        if (k == 1) return 0;
    }
}

__device__ __forceinline__ bool stage_buckets(Stager &sg, ItemInfo x, const SliceDesc *d, uint32_t c_lo, uint32_t k,
                                              BatchHeader *hdr)
{
    const uint32_t core = x.core, m = core_buckets(d, core);
    const uint64_t wait_ns = hdr->wait_ns;
    for (uint32_t j = 0; j < m; j += k) {
        const uint32_t kk = min(k, m - j), off = j * d->bkt_w;
        const BucketRange r(d, c_lo + j, kk);
        const uint32_t n = r.hits(d);
        if (n == 0) continue;
        if (!sg.wait_free(hdr, wait_ns)) return false;
        x.rank_lo = __ldg(d->bkt_off + r.b_lo);
        x.off = off, x.core = min(kk * d->bkt_w, core - off);
        x.lo_t = r.lead * d->bkt_w, x.span = (r.b_hi - r.b_lo) * d->bkt_w;
        sg.hand_over(x, n);
        if (lane_id() == 0 && CHECK(7, (uint64_t)x.rank_lo + n, d->n_hits + 1))
            bulk_g2s(sg.stage, d->tbuf + x.rank_lo, n * 16u, sg.full);
    }
    if (!sg.wait_free(hdr, wait_ns)) return false;
    x.mode = kItemEnd;
    sg.hand_over(x, 0);
    return true;
}

template <int CAP, int NC, bool SMEM_DT, bool EXT, bool DENSE>
__global__ void __launch_bounds__(NC + 32, (CAP <= 1024 ? 4 : CAP <= 2048 ? 2 : 1)) k_tile(BatchHeader *__restrict__ hdr,
                                                                          const SliceDesc *__restrict__ desc,
                                                                          uint32_t max_pmt)
{
    constexpr uint32_t NW = NC / 32;
    using C = TileCtx<CAP, NC, SMEM_DT, EXT>;
    using L = typename C::L;
    __shared__ uint64_t full_bar, empty_bar;
    __shared__ ItemInfo info;
    __shared__ uint2 pieces[kMaxPieces], runs[32 * kStageRuns];

    C cx;
    cx.pp = (max_pmt + 7) & ~7u;
    cx.dt_g = nullptr;
    cx.P = 0;
    cx.tab = (uint32_t)L::tab(max_pmt);

    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    if (tid == 0) {
        mbar_init(&full_bar, 1);
        mbar_init(&empty_bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    wait_for_previous_kernel();
    let_next_kernel_in();

    const uint32_t n_slices = hdr->n_slices, n_items = hdr->n_items;
    const uint64_t wait_ns = hdr->wait_ns;

    if (warp == NW) {
        // test control: stage nothing, so that the consumers' first wait
        // runs out (no copy is ever in flight)
        if (hdr->stall) return;
        // ------------------------------------------------ producer warp
        // The next item is dequeued and its per-PMT runs looked up before
        // waiting for a free buffer, so those global loads overlap the wait.
        uint32_t s = 0;
        bool bad = false;
        const SliceDesc *d = nullptr;
        constexpr int R = kStageRuns;              // PMTs per lane kept in registers
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(&hdr->queue, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        Stager sg{&full_bar, &empty_bar, &info, cx.stage(), 0u};
        for (;;) {
#ifdef TRIG_PHASE_STATS
            const long long tp0 = clock64();
#endif
            uint32_t g = 0, P = 0, mode = kItemSkip, lo_t = 0, span = 0, core = 0;
            uint32_t ra[R], rl[R];                  // hit indices are below 2^32 - 16
            uint32_t tot = 0, rlo = 0, c_lo = 0, piece = 0;
            bool wide = false;
            if (item < n_items) {
                // items arrive in increasing order: walk the slice index forward
                if (d == nullptr || item < d->item0) s = find_slice_by_item(desc, n_slices, item), d = nullptr;
                while (s + 1 < n_slices && desc[s + 1].item0 <= item) ++s, d = nullptr;
                if (d == nullptr) {
                    d = &desc[s];
                    bad = (d->stats->flags & (TRIG_FLAG_BAD_PMT | TRIG_FLAG_UNSORTED | TRIG_FLAG_OUT_OF_RANGE)) != 0;
                }
                g = item - d->item0;
                P = d->n_pmt;
                wide = d->wide != 0;
                core = (uint32_t)min(d->tile_w, d->slice_ns - (int64_t)g * d->tile_w);
                if (wide) {
                    // one contiguous range of the bucketed copy: the core
                    // buckets and hh buckets of halo on each side
                    c_lo = d->bkt_lead + g * d->bkt_per_tile;
                    const BucketRange r(d, c_lo, d->bkt_per_tile);
                    lo_t = r.lead * d->bkt_w;
                    span = (r.b_hi - r.b_lo) * d->bkt_w;
                    if (!bad) {
                        rlo = __ldg(d->bkt_off + r.b_lo);
                        tot = r.hits(d);
                        if (tot > (uint32_t)CAP) piece = piece_buckets(d, c_lo, core, CAP);
                    }
                } else {
                    // the PMTs' runs [lb(B_g - H), lb(B_{g+1} + H)), P <= 32 R
                    const uint32_t *elo = d->edge + (size_t)(2u * g) * P;
                    const uint32_t *ehi = d->edge + (size_t)(2u * (g + d->edge_a) + 1u) * P;
                    const uint64_t *poff = d->pmt_off;
                    lo_t = d->halo;
                    span = (uint32_t)d->tile_w + 2u * d->halo;
                    if (!bad) {
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const uint32_t p = r * 32 + lane;
                            uint32_t a = 0, e = 0, sp_ = 0, ep_ = 0;
                            if (p < P) {
                                a = __ldg(elo + p);
                                e = __ldg(ehi + p);
                                sp_ = (uint32_t)__ldg(poff + p);
                                ep_ = (uint32_t)__ldg(poff + p + 1);
                                a = min(max(a, sp_), ep_);
                                e = min(max(e, a), ep_);
                            }
                            ra[r] = a;
                            rl[r] = e - a;
                            tot += e - a;
                            rlo += a - sp_;
                        }
                    }
                    tot = __reduce_add_sync(0xffffffffu, tot);
                    rlo = __reduce_add_sync(0xffffffffu, rlo);
                }
                mode = bad || tot == 0                ? kItemSkip
                       : tot <= (uint32_t)CAP    ? kItemTile
                       : wide && piece == 0      ? kItemDefer
                                                 : kItemPiece;
            }
            uint32_t next = 0;
            if (item < n_items) {
                if (lane == 0) next = atomicAdd(&hdr->queue, 1u);
                next = __shfl_sync(0xffffffffu, next, 0);
            }
#ifdef TRIG_PHASE_STATS
            if (lane == 0) PHASE_ADD(kPhProdItem, clock64() - tp0);
#endif
            if (item >= n_items) {
                if (sg.wait_free(hdr, wait_ns)) sg.hand_over(ItemInfo{-1}, 0);
                break;
            }
            const ItemInfo x{(int32_t)item, s, g, 0, rlo, mode, 0, core, lo_t, span};
            if (mode == kItemPiece && wide) {
                if (!stage_buckets(sg, x, d, c_lo, piece, hdr)) break;
            } else if (mode == kItemPiece) {
#pragma unroll
                for (int r = 0; r < R; ++r) runs[r * 32 + lane] = make_uint2(ra[r], ra[r] + rl[r]);
                __syncwarp();
                if (!stage_pieces(sg, x, CAP, kCrowdCap<CAP, NC>, d, runs, pieces, hdr)) break;
            } else {
                if (!sg.wait_free(hdr, wait_ns)) break;
                sg.hand_over(x, mode == kItemTile ? tot : 0u);
                if (mode == kItemTile && wide) {
                    if (lane == 0 && CHECK(7, (uint64_t)rlo + tot, d->n_hits + 1))
                        bulk_g2s(cx.stage(), d->tbuf + rlo, tot * 16u, &full_bar);
                } else if (mode == kItemTile) {
                    uint32_t dst = 0;
#pragma unroll
                    for (int r = 0; r < R; ++r) sg.copy_run(d->hits, d->n_hits, ra[r], rl[r], CAP, dst);
                }
            }
#ifdef TRIG_PHASE_STATS
            if (lane == 0) PHASE_ADD(kPhProdTotal, clock64() - tp0);
#endif
            item = next;
        }
        return;
    }

    // ---------------------------------------------------- consumer warps
    // the tile pass expects zero bucket counts, mask and cells (and leaves them so)
    for (uint32_t i = tid; i < (uint32_t)L::NBK; i += NC) cx.cnt()[i] = 0;
    for (uint32_t i = tid; i < (uint32_t)CAP / 32; i += NC) cx.mask()[i] = 0;
    for (uint32_t i = tid; i < L::kCells / 16; i += NC) cx.cells()[i] = 0;
    cons_sync<NC>();
    const SliceDesc *loaded = nullptr;
    // the slice's trigger parameters live in shared memory (written by one
    // thread when the slice changes), keeping registers for the tile phases
    __shared__ TrigParams tp;
    // the loaded slice's tile width, t0 and merged rank of its first owned
    // hit, also kept in shared memory
    __shared__ int64_t sl[3];
    // the tables of a slice's detector (kept while the next slice has the
    // same) and its parameters
    auto load_slice = [&](const SliceDesc &d) {
        if (cx.dt_g != d.dt) {
            const uint32_t P = d.n_pmt;
            for (uint32_t p = tid; p < P; p += NC) {
                cx.floor_s()[p] = d.floor[p];
                cx.dmax_s()[p] = d.dmax_row[p];
            }
            // seed rule 1: the PMT relation above a dt that leaves it room
            const bool pack = EXT && SMEM_DT && d.rel_in_dt;
            if (SMEM_DT)
                for (uint32_t p = warp; p < P; p += NW)
                    for (uint32_t q = lane; q < P; q += 32) {
                        uint32_t v = d.dt[p * P + q];
                        if (pack) v |= (uint32_t)d.rel[p * P + q] << kRelShift;
                        cx.dt_s()[p * (kDtRow / 2) + q] = (uint16_t)v;
                    }
            cx.dt_g = d.dt;
            cx.P = P;
        }
        loaded = &d;
        if (tid == 0) {
            tp.H = d.halo;
            tp.win_half = d.win_half;
            tp.tau = d.tau;
            tp.q_seed = d.q_seed;
            tp.threshold = d.threshold;
            tp.l0_hits = d.l0_hits;
            tp.l0_window = d.l0_window;
            tp.l0_distinct = d.l0_distinct;
            tp.seed_rule = d.seed_rule;
            tp.sc_w = d.sc_w;
            tp.fc_w = d.fc_w;
            tp.afc_w = d.afc_w;
            tp.count_distinct = d.count_distinct;
            tp.dt_mask = EXT && SMEM_DT && d.rel_in_dt ? (1u << kRelShift) - 1u : 0xffffu;
            tp.rel = d.rel;
            tp.dbg_merged = d.dbg_merged;
            tp.dbg_seedcnt = d.dbg_seedcnt;
            sl[0] = d.tile_w;
            sl[1] = d.t0;
            sl[2] = (int64_t)d.dbg_rank0;
        }
    };
    // while the first tile is looked up and copied: the slice it is in if the
    // blocks take the first items in turn
    if (n_items) load_slice(desc[find_slice_by_item(desc, n_slices, min(blockIdx.x, n_items - 1u))]);
    // the tile whose pieces are coming: its fired seeds so far, where they
    // start, whether a piece was seen, and its seeds (thread 0 writes after a
    // pass; the next tile's barrier publishes it)
    __shared__ uint32_t pc[4];
    if (tid < 4) pc[tid] = 0;
    // the block's tiles that are put off, the last one first: the item before
    // each stands in its tile_nfired
    __shared__ uint32_t deferred;
    if (tid == 0) deferred = kNoItem;
    bool done = false;
    for (uint32_t it = 0;; ++it) {
        // every thread waits (bounded) for the staged tile; the barrier
        // ANDs their results, so the block never splits on a timeout
#ifdef TRIG_PHASE_STATS
        const long long tw0 = clock64();
        uint32_t cr = 0;
        const bool cwait_ok = mbar_wait(&full_bar, it & 1u, wait_ns, &cr);
        if (tid == 0) {
            PHASE_ADD(kPhConsWait, clock64() - tw0);
            PHASE_ADD(kPhConsWaitRounds, cr);
            PHASE_ADD(kPhTiles, 1);
        }
#else
        const bool cwait_ok = mbar_wait(&full_bar, it & 1u, wait_ns);
#endif
        if (!named_sync_and(kBarCons, NC, cwait_ok)) {
            if (tid == 0) atomicOr(&hdr->err, TRIG_FLAG_TIMEOUT);
            break;
        }
        const ItemInfo &inf = info;      // stable until this buffer is released
        if (inf.item < 0) {
            done = true;
            break;
        }
        const SliceDesc &d = desc[inf.slice];
        if (&d != loaded) {
            cons_sync<NC>();
            load_slice(d);
            cons_sync<NC>();
        }
        if (inf.mode == kItemSkip || inf.mode == kItemEnd || inf.mode == kItemDefer) {
            if (tid == 0) {
                if (inf.mode == kItemDefer) {
                    d.tile_nfired[inf.g] = deferred;
                    deferred = (uint32_t)inf.item;
                } else {
                    d.tile_nfired[inf.g] = pc[0];
                    d.tile_rank[inf.g] = pc[1];
                    if (pc[3]) atomicAdd(reinterpret_cast<unsigned long long *>(&d.stats->n_seeds), (unsigned long long)pc[3]);
                }
                pc[0] = pc[1] = pc[2] = pc[3] = 0;
            }
        } else {
            const uint32_t g = inf.g, n_st = inf.n, rank_lo = inf.rank_lo, span = inf.span, lo_t = inf.lo_t;
            const uint32_t hi_t = lo_t + inf.core;
            const bool piece = inf.mode == kItemPiece;
            // the staged range starts lo_t (>= H) before the core
            const int64_t tb = sl[1] + (int64_t)g * sl[0] + (int64_t)inf.off - (int64_t)lo_t;
            // a tile's (or its first piece's) fired seeds go to the merged
            // rank of its first core hit, rank_lo + c0; the other pieces'
            // follow them.  The pass hands the buffer back as soon as it has
            // read it (inf is not read after that)
            const bool seen = pc[2] != 0;
            const size_t at = seen ? pc[1] + pc[0] : rank_lo;
            const CoreOut co = tile_pass<CAP, NC, SMEM_DT, EXT, DENSE>(cx, cx.stage(), n_st, tb, span, lo_t, hi_t, tp, d.stage + at,
                                                                       d.wrank + 2 * at, !seen, rank_lo,
                                                                       (int64_t)rank_lo - sl[2], &empty_bar);
            const uint32_t tile_rank = rank_lo + co.c0;
            if (tid == 0 && CHECK(14, (uint64_t)tile_rank + co.n_fired, d.n_hits + 1) && CHECK(15, g, d.n_tiles)) {
                if (!piece) {
                    d.tile_nfired[g] = co.n_fired;
                    d.tile_rank[g] = tile_rank;
                    atomicAdd(reinterpret_cast<unsigned long long *>(&d.stats->n_seeds), (unsigned long long)co.n_seeds);
                } else {
                    if (!pc[2]) pc[1] = tile_rank, pc[2] = 1;
                    pc[0] += co.n_fired;
                    pc[3] += co.n_seeds;
                }
            }
            continue;
        }
        // release the buffer to the producer: order our generic-proxy
        // accesses before its next bulk copy into the same buffer
        fence_proxy_async_smem();
        cons_sync<NC>();
        if (tid == 0) mbar_arrive(&empty_bar);
    }
    if (!done) return;                   // a wait ran out
    // the tiles put off: out of the loop above, whose registers they would take
    for (uint32_t item; (item = deferred) != kNoItem; cons_sync<NC>()) {
        const SliceDesc &d = desc[find_slice_by_item(desc, n_slices, item)];
        cons_sync<NC>();                 // every thread has read `deferred`
        if (&d != loaded) load_slice(d);
        if (tid == 0) deferred = d.tile_nfired[item - d.item0];
        cons_sync<NC>();
        if constexpr (EXT) put_off_tile<CAP, NC, SMEM_DT, EXT, DENSE>(cx, d, item - d.item0, tp);
        else put_off_call<CAP, NC, SMEM_DT, EXT, DENSE>(cx.P, cx.tab, cx.pp, cx.dt_g, &d, item - d.item0, &tp);
    }
}

// ------------------------------------------------------------ window ranks

// Where the first hit of PMT p's stream at or past time x can be, narrowed by
// the tile edges the structure pass recorded: x between the edges B_g - H and
// B_{g+1} - H lies between the PMT's offsets there, so a binary search covers
// a handful of hits.  Outside the edges the first or last one bounds it.
__device__ __forceinline__ void rank_range(const SliceDesc &d, uint32_t p, int64_t x, uint32_t sp, uint32_t ep, uint32_t &lo,
                                           uint32_t &hi)
{
    const int64_t rel = x - (d.t0 - (int64_t)d.halo);
    lo = sp;
    hi = ep;
    if (rel >= 0) {
        const int64_t g = min(rel / d.tile_w, (int64_t)d.n_tiles);
        const uint32_t *at = d.edge + (size_t)(2 * g) * d.n_pmt + p;
        lo = max(lo, min(at[0], ep));
        if (g < (int64_t)d.n_tiles) hi = min(hi, max(at[2 * (size_t)d.n_pmt], lo));
    } else if (d.n_tiles) {
        hi = min(hi, max(d.edge[p], lo));
    }
}

// That first hit's index.
__device__ __forceinline__ uint64_t rank_in_pmt(const SliceDesc &d, uint32_t p, int64_t x, uint64_t sp, uint64_t ep)
{
    uint32_t lo, hi;
    rank_range(d, p, x, (uint32_t)sp, (uint32_t)ep, lo, hi);
    return lb_time(d.hits, lo, hi, x);
}

// Merged rank of time x (the hits of the submission with t < x), by the
// warp: per-PMT searches, a lane's four side by side (one after the other
// they were the longest chain behind a slice's windows), or for a wide slice
// the bucket offsets plus the edge bucket's hits below x.
__device__ __noinline__ uint64_t warp_rank_of(const SliceDesc &d, int64_t x)
{
    const uint32_t lane = lane_id();
    uint64_t r = 0;
    if (d.wide) {
        const uint32_t bx = bkt_index(d, x);
        const uint32_t e0 = d.bkt_off[bx], e1 = d.bkt_off[bx + 1];
        if (lane == 0) r = e0;
        for (uint32_t j = e0 + lane; j < e1; j += 32) r += d.tbuf[j].t_ns < x;
    } else {
        constexpr uint32_t R = (kWideMinPmt + 30) / 32;
        uint32_t lo[R], hi[R], own = 0;
        bool more = false;
#pragma unroll
        for (uint32_t k = 0; k < R; ++k) {
            const uint32_t p = k * 32 + lane;
            lo[k] = hi[k] = 0;
            if (p < d.n_pmt) {
                const uint32_t sp = (uint32_t)d.pmt_off[p];
                rank_range(d, p, x, sp, (uint32_t)d.pmt_off[p + 1], lo[k], hi[k]);
                own -= sp;
            }
            more |= lo[k] < hi[k];
        }
        while (more) {
            int64_t t[R];
#pragma unroll
            for (uint32_t k = 0; k < R; ++k)
                if (lo[k] < hi[k]) t[k] = d.hits[lo[k] + ((hi[k] - lo[k]) >> 1)].t_ns;
            more = false;
#pragma unroll
            for (uint32_t k = 0; k < R; ++k) {
                if (lo[k] >= hi[k]) continue;
                const uint32_t mid = lo[k] + ((hi[k] - lo[k]) >> 1);
                if (t[k] < x) lo[k] = mid + 1u;
                else hi[k] = mid;
                more |= lo[k] < hi[k];
            }
        }
#pragma unroll
        for (uint32_t k = 0; k < R; ++k) own += lo[k];
        r = own;                        // the lane's sum: at most its hits, so below 2^32
    }
    return warp_sum_u64(r);
}

// ----------------------------------------------------------------- k_final

// What the windows need to know of a run of consecutive triggers of a slice.
// A trigger is a head (starts a window) unless it lies within 2h + 1 ns of
// the slice's trigger before it (windows [t - h, t + h] merge while
// lo_next <= hi_cur + 1); whether a run's first trigger is one depends on
// what comes before, so it is left out of `heads`.
struct FinRun {
    uint32_t n;             // triggers
    uint32_t heads;         // heads after the first trigger
    uint32_t k;             // the last of them: its place in the run,
    uint32_t r;             //   and the merged rank of its window's first hit
    uint32_t r_first;       // the same rank for the run's first trigger
    uint32_t r_last;        // the rank one past the window of the run's last trigger
    int64_t t_first, t_last, t_head;
};

// a, then b.
__device__ __forceinline__ FinRun fin_join(const FinRun &a, const FinRun &b, int64_t gap)
{
    if (a.n == 0) return b;
    if (b.n == 0) return a;
    const bool bh = b.t_first - a.t_last > gap;
    FinRun o;
    o.n = a.n + b.n;
    o.heads = a.heads + b.heads + (bh ? 1u : 0u);
    o.k = b.heads ? a.n + b.k : bh ? a.n : a.k;
    o.r = b.heads ? b.r : bh ? b.r_first : a.r;
    o.t_head = b.heads ? b.t_head : bh ? b.t_first : a.t_head;
    o.r_first = a.r_first;
    o.r_last = b.r_last;
    o.t_first = a.t_first;
    o.t_last = b.t_last;
    return o;
}

template <bool UP>
__device__ __forceinline__ FinRun fin_shfl(const FinRun &a, uint32_t off)
{
    auto mv = [&](auto x) {
        return UP ? __shfl_up_sync(0xffffffffu, x, off) : __shfl_down_sync(0xffffffffu, x, off);
    };
    FinRun o;
    o.n = mv(a.n), o.heads = mv(a.heads), o.k = mv(a.k), o.r = mv(a.r), o.r_first = mv(a.r_first), o.r_last = mv(a.r_last);
    o.t_first = mv(a.t_first), o.t_last = mv(a.t_last), o.t_head = mv(a.t_head);
    return o;
}

// What a chunk has published: flag 1, its own run (run[0]); 2, the slice's
// run up to its end (run[1]; a reader may still be taking run[0]).
struct FinState {
    uint32_t flag, pad;
    FinRun run[2];
};
static_assert(sizeof(FinState) == kFinStateBytes, "sized by the planner");

__device__ __forceinline__ void fin_publish(FinState *st, const FinRun &run, uint32_t flag)
{
    st->run[flag - 1u] = run;
    __threadfence();
    atomicExch(&st->flag, flag);
}

__device__ __forceinline__ FinRun fin_load(const FinState *st, uint32_t flag)
{
    FinRun r;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(&st->run[flag - 1u]);
    uint32_t *dst = reinterpret_cast<uint32_t *>(&r);
#pragma unroll
    for (uint32_t i = 0; i < sizeof(FinRun) / 4; ++i) dst[i] = __ldcg(src + i);
    return r;
}

__device__ __forceinline__ int32_t status_of(uint32_t f)
{
    if (f & (TRIG_FLAG_BAD_PMT | TRIG_FLAG_UNSORTED | TRIG_FLAG_OUT_OF_RANGE)) return TRIG_EINVAL;
    if (f & TRIG_FLAG_TIMEOUT) return TRIG_ETIMEOUT;
    if (f & (TRIG_FLAG_TILE_FULL | TRIG_FLAG_TRIG_FULL | TRIG_FLAG_WIN_FULL | TRIG_FLAG_EV_FULL)) return TRIG_ECAPACITY;
    return TRIG_OK;
}

// One window (by the lanes that hold one, the whole warp calling): the edge
// ranks the tile pass could not read off its staged keys are searched for.
__device__ __forceinline__ void fin_window(const SliceDesc &d, bool have, uint64_t w, int64_t lo, int64_t hi, uint32_t r_lo,
                                           uint32_t r_hi, uint32_t n_trig)
{
    const uint32_t lane = lane_id();
    have = have && w < d.win_cap;
    for (uint32_t m = __ballot_sync(0xffffffffu, have && r_lo == kRankUnknown); m; m &= m - 1u) {
        const uint32_t l = __ffs(m) - 1;
        const uint64_t r = warp_rank_of(d, __shfl_sync(0xffffffffu, lo, l));
        if (lane == l) r_lo = (uint32_t)r;
    }
    for (uint32_t m = __ballot_sync(0xffffffffu, have && r_hi == kRankUnknown); m; m &= m - 1u) {
        const uint32_t l = __ffs(m) - 1;
        const uint64_t r = warp_rank_of(d, __shfl_sync(0xffffffffu, hi, l) + 1);
        if (lane == l) r_hi = (uint32_t)r;
    }
    if (!have) return;
    trig_window out;
    out.lo_ns = lo;
    out.hi_ns = hi;
    out.n_hits = r_hi - r_lo;
    out.n_triggers = n_trig;
    d.windows[w] = out;
    if (d.ev && d.ev_cap) d.win_rlo[w] = r_lo;
}

// Stream compaction of the fired seeds and the window merge, in one pass
// over the tiles' seeds: a block takes kFinTiles tiles of a slice at a time
// (in order, by a ticket), reduces their seeds to a FinRun, publishes it,
// gets the run of everything before from the published ones (decoupled
// look-back, after Merrill and Garland, "Single-pass Parallel Prefix Scan with
// Decoupled Look-back", NVIDIA 2016: the tickets' order makes the blocks it
// waits for running ones; the wait is bounded like the tile pass's), then copies the seeds to the
// dense list and writes each window from the head that follows it.  One
// launch where a scan, a copy, a scan, a window pass, a count pass and a
// status pass were six, each reading what the one before had written: 14 us
// against 36 behind one 320 k-hit slice, 0.27 ms against 0.44 behind 64
// slices of 12 M triggers.  Bound by the latency of its chain (ticket, tile
// counts, two reads of the seeds around the look-back).
constexpr uint32_t kFinThreads = 256;
constexpr uint32_t kFinUnroll = 2;          // loads of a warp's pass in flight (four spill)

__global__ void __launch_bounds__(kFinThreads, 3) k_final(BatchHeader *__restrict__ hdr, const SliceDesc *__restrict__ desc)
{
    constexpr uint32_t NW = kFinThreads / 32;
    __shared__ uint32_t s_chunk, s_err, s_off[kFinTiles + 1], s_rank[kFinTiles];
    __shared__ FinRun s_run[NW], s_before;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5, lt = (1u << lane) - 1u;
    wait_for_previous_kernel();
    const uint32_t n_slices = hdr->n_slices, n_chunks = hdr->n_fin;
    for (;;) {
        if (tid == 0) {
            s_chunk = atomicAdd(&hdr->fin_queue, 1u);
            s_err = __ldcg(&hdr->err);
        }
        __syncthreads();
        const uint32_t c = s_chunk;
        if (c >= n_chunks) return;
        uint32_t s = 0;
        for (uint32_t hi = n_slices; hi - s > 1;) {           // largest s with fin0 <= c
            const uint32_t mid = (s + hi) >> 1;
            if (desc[mid].fin0 <= c) s = mid; else hi = mid;
        }
        const SliceDesc &d = desc[s];
        const uint32_t ci = c - d.fin0, g0 = ci * kFinTiles;
        const bool last = g0 + kFinTiles >= d.n_tiles;
        // the tile pass gave up: its per-tile outputs are not valid
        if (s_err) {
            if (last && tid == 0) {
                const uint32_t f = d.stats->flags | s_err;
                d.stats->flags = f;
                d.stats->status = status_of(f);
            }
            __syncthreads();
            continue;
        }
        const int64_t gap = 2 * (int64_t)d.win_half + 1, half = d.win_half;
        if (warp == 0) {
            const uint32_t g = g0 + lane;
            const uint32_t nf = lane < kFinTiles && g < d.n_tiles ? d.tile_nfired[g] : 0u;
            if (lane < kFinTiles) s_rank[lane] = g < d.n_tiles ? d.tile_rank[g] : 0u;
            const uint32_t incl = warp_incl_scan(nf);
            if (lane < kFinTiles) s_off[lane] = incl - nf;
            if (lane == 31) s_off[kFinTiles] = incl;
        }
        __syncthreads();
        const uint32_t n = s_off[kFinTiles];
        // the chunk's seed f: in the last tile with s_off <= f
        auto src_of = [&](uint32_t f) {
            uint32_t g = 0;
#pragma unroll
            for (uint32_t step = kFinTiles / 2; step; step >>= 1)
                if (s_off[g + step] <= f) g += step;
            return s_rank[g] + (f - s_off[g]);
        };
        // each warp takes a contiguous share
        const uint32_t share = ((n + NW - 1) / NW + 31u) & ~31u;
        const uint32_t fa = min(n, warp * share), fb = min(n, fa + share);
        FinRun run{};
        uint32_t src_h = 0;
        for (uint32_t x = fa; x < fb; x += 32 * kFinUnroll) {
            uint32_t src[kFinUnroll];
            int64_t tt[kFinUnroll];
#pragma unroll
            for (uint32_t u = 0; u < kFinUnroll; ++u) {
                src[u] = src_of(min(x + 32 * u + lane, fb - 1u));
                tt[u] = d.stage[src[u]].t_ns;
            }
#pragma unroll
            for (uint32_t u = 0; u < kFinUnroll; ++u) {
                const uint32_t f0 = x + 32 * u, f = f0 + lane;
                if (f0 >= fb) break;
                const int64_t t = tt[u];
                int64_t tp = __shfl_up_sync(0xffffffffu, t, 1);
                if (lane == 0) tp = run.t_last;
                const bool head = f < fb && f > fa && t - tp > gap;
                const uint32_t m = __ballot_sync(0xffffffffu, head);
                if (m) {
                    const uint32_t l = 31u - __clz(m);
                    run.heads += __popc(m);
                    run.k = f0 + l - fa;
                    src_h = __shfl_sync(0xffffffffu, src[u], l);
                    run.t_head = __shfl_sync(0xffffffffu, t, l);
                }
                if (f0 == fa) run.t_first = __shfl_sync(0xffffffffu, t, 0);
                run.t_last = __shfl_sync(0xffffffffu, t, 31);
            }
        }
        if (fa < fb) {
            run.r_first = d.wrank[2 * (size_t)src_of(fa)];
            run.r_last = d.wrank[2 * (size_t)src_of(fb - 1u) + 1];
            if (run.heads) run.r = d.wrank[2 * (size_t)src_h];
        }
        run.n = fb - fa;
        if (lane == 0) s_run[warp] = run;
        __syncthreads();
        if (warp == 0) {
            // runs of the warps before each warp, and of the whole chunk
            FinRun a{};
            if (lane < NW) a = s_run[lane];
            for (uint32_t off = 1; off < NW; off <<= 1) {
                const FinRun b = fin_shfl<true>(a, off);
                if (lane >= off) a = fin_join(b, a, gap);
            }
            FinState *st = reinterpret_cast<FinState *>(d.fin) + ci;
            if (lane == NW - 1) {
                s_before = a;
                if (!last) fin_publish(st, a, ci == 0 ? 2u : 1u);
            }
            __syncwarp();
            const FinRun all = s_before;
            a = fin_shfl<true>(a, 1);
            if (lane == 0) a = FinRun{};
            // look back: the nearest chunk with the slice's run up to it,
            // all later ones with their own
            FinRun before{};
            if (ci > 0) {
                const FinState *mine = lane < ci ? st - 1 - lane : nullptr;
                const uint64_t t0 = global_ns();
                uint32_t to = 0, f;
                for (;;) {
                    f = 0;
                    if (mine) f = __ldcg(&mine->flag);
                    const uint32_t full = __ballot_sync(0xffffffffu, f == 2u), any = __ballot_sync(0xffffffffu, f != 0u);
                    if (full) {
                        to = __ffs(full) - 1u;
                        if ((any & ((1u << to) - 1u)) == ((1u << to) - 1u)) break;
                    }
                    const bool out = __shfl_sync(0xffffffffu, (int)(global_ns() - t0 > hdr->wait_ns), 0);
                    if (out) {
                        if (lane == 0) atomicOr(&hdr->err, TRIG_FLAG_TIMEOUT);
                        to = 0xffffffffu;
                        break;
                    }
                }
                __threadfence();                // the flags before what they stand for
                if (to != 0xffffffffu && lane <= to) before = fin_load(mine, f);
                for (uint32_t off = 1; off < 32; off <<= 1) {
                    const FinRun b = fin_shfl<false>(before, off);
                    if (lane + off < 32) before = fin_join(b, before, gap);
                }
                if (lane == 0 && !last) fin_publish(st, fin_join(before, all, gap), 2u);
            }
            FinRun p;                                  // lane 0's for every lane
            {
                const uint32_t *x = reinterpret_cast<const uint32_t *>(&before);
                uint32_t *y = reinterpret_cast<uint32_t *>(&p);
#pragma unroll
                for (uint32_t i = 0; i < sizeof(FinRun) / 4; ++i) y[i] = __shfl_sync(0xffffffffu, x[i], 0);
            }
            if (lane < NW) s_run[lane] = fin_join(p, a, gap);
            if (last) {
                // the slice's last window, its counters and status
                const FinRun z = fin_join(p, all, gap);
                const bool inner = z.heads > 0;
                fin_window(d, lane == 0 && z.n > 0, z.heads, (inner ? z.t_head : z.t_first) - half, z.t_last + half,
                           inner ? z.r : z.r_first, z.r_last, z.n - (inner ? z.k : 0u));
                if (lane == 0) {
                    // (a wait that ran out before: the sums are not valid)
                    const uint32_t err = __ldcg(&hdr->err), nt = err ? 0u : z.n;
                    const uint64_t nw = nt ? (uint64_t)z.heads + 1u : 0u;
                    uint32_t f = d.stats->flags | err;
                    if (nt > d.trig_cap) f |= TRIG_FLAG_TRIG_FULL;
                    if (nw > d.win_cap) f |= TRIG_FLAG_WIN_FULL;
                    d.stats->n_triggers = nt;
                    d.stats->n_windows = nw;
                    d.stats->flags = f;
                    d.stats->status = status_of(f);
                }
            }
        }
        __syncthreads();
        // copy the share's seeds and write the windows that its heads close
        FinRun p = s_run[warp];
        const uint2 *wr = reinterpret_cast<const uint2 *>(d.wrank);
        uint32_t rhi_last = p.r_last;
        for (uint32_t x = fa; x < fb; x += 32 * kFinUnroll) {
            int4 vv[kFinUnroll];
            uint2 ww[kFinUnroll];
#pragma unroll
            for (uint32_t u = 0; u < kFinUnroll; ++u) {
                const uint32_t src = src_of(min(x + 32 * u + lane, fb - 1u));
                vv[u] = *reinterpret_cast<const int4 *>(d.stage + src);
                ww[u] = wr[src];
            }
#pragma unroll
            for (uint32_t u = 0; u < kFinUnroll; ++u) {
                const uint32_t f0 = x + 32 * u, f = f0 + lane;
                if (f0 >= fb) break;
                const int4 v = vv[u];
                const uint2 rk = ww[u];          // ranks of the window's first hit, and one past it
                const uint64_t o = (uint64_t)p.n + lane;
                if (f < fb && o < d.trig_cap) *reinterpret_cast<int4 *>(d.triggers + o) = v;
                const int64_t t = (int64_t)(((uint64_t)(uint32_t)v.y << 32) | (uint32_t)v.x);
                int64_t tp = __shfl_up_sync(0xffffffffu, t, 1);
                uint32_t r_hi = __shfl_up_sync(0xffffffffu, rk.y, 1);
                if (lane == 0) tp = p.t_last, r_hi = rhi_last;
                const bool first = p.n == 0 && lane == 0;            // of the slice
                const bool head = f < fb && (first || t - tp > gap);
                const uint32_t m = __ballot_sync(0xffffffffu, head);
                if (m) {
                    const uint32_t r = rk.x;
                    // the head before this one, in this step or before it
                    const uint32_t before = m & lt, l = before ? 31u - __clz(before) : 0u;
                    const int64_t th = __shfl_sync(0xffffffffu, t, l);
                    const uint32_t rh = __shfl_sync(0xffffffffu, r, l);
                    const bool inner = p.heads > 0;
                    const int64_t t_h = before ? th : inner ? p.t_head : p.t_first;
                    const uint32_t r_h = before ? rh : inner ? p.r : p.r_first;
                    const uint32_t k_h = before ? p.n + l : inner ? p.k : 0u;
                    const bool close = head && !first;
                    // heads before this one, less the slice's first
                    const uint32_t w = p.n == 0 ? __popc(before) - 1u : p.heads + __popc(before);
                    fin_window(d, close, w, t_h - half, tp + half, r_h, r_hi, (uint32_t)o - k_h);
                    const uint32_t e = 31u - __clz(m), ne = __popc(m) - (p.n == 0 ? 1u : 0u);
                    const int64_t te = __shfl_sync(0xffffffffu, t, e);
                    const uint32_t re = __shfl_sync(0xffffffffu, r, e);
                    if (p.n == 0) p.t_first = __shfl_sync(0xffffffffu, t, 0), p.r_first = __shfl_sync(0xffffffffu, r, 0);
                    if (ne) p.t_head = te, p.r = re, p.k = p.n + e;
                    p.heads += ne;
                }
                p.t_last = __shfl_sync(0xffffffffu, t, 31);
                rhi_last = __shfl_sync(0xffffffffu, rk.y, 31);
                p.n += min(32u, fb - f0);
            }
        }
        __syncthreads();
    }
}

// ----------------------------------------------------- event extraction

// The slice's leading halo (t < t0) and trailing halo (t >= t0 + S) in
// merged order at the two ends of its merged stream (the tile pass writes
// the owned hits between them, at their merged ranks).  One block per
// slice; each halo is gathered into shared memory as keys relative to its
// start and ranked by counting.  More than TRIG_EV_HALO_MAX hits in a halo
// sets TRIG_FLAG_EV_FULL.
constexpr uint32_t kEvHaloThreads = 1024;

__device__ void ev_halo_side(const SliceDesc &d, bool lead, uint64_t *keys, uint32_t *psum, int64_t base, int64_t t_cut)
{
    const uint32_t tid = threadIdx.x, P = d.n_pmt;
    const trig_hit *hits = d.hits;
    const uint64_t *poff = d.pmt_off;
    // the first hit past the cut, between the tile edges around it where the
    // structure pass recorded them (about 4 loads in a row instead of 16)
    auto halo_cut = [&](uint32_t p) {
        return d.wide ? lb_time(hits, poff[p], poff[p + 1], t_cut) : rank_in_pmt(d, p, t_cut, poff[p], poff[p + 1]);
    };
    // per-PMT counts of the halo hits (each thread a contiguous run of PMTs)
    const uint32_t per = (P + kEvHaloThreads - 1) / kEvHaloThreads;
    const uint32_t p0 = min(P, tid * per), p1 = min(P, p0 + per);
    uint32_t local = 0;
    for (uint32_t p = p0; p < p1; ++p) {
        const uint64_t a = halo_cut(p);
        local += (uint32_t)(lead ? a - poff[p] : poff[p + 1] - a);
    }
    // exclusive block scan of the per-thread counts
    psum[tid] = local;
    __syncthreads();
    for (uint32_t off = 1; off < kEvHaloThreads; off <<= 1) {
        const uint32_t v = tid >= off ? psum[tid - off] : 0u;
        __syncthreads();
        psum[tid] += v;
        __syncthreads();
    }
    const uint32_t total = psum[kEvHaloThreads - 1];
    uint32_t at = psum[tid] - local;
    __syncthreads();
    if (total > TRIG_EV_HALO_MAX) {
        if (tid == 0) report(d, TRIG_FLAG_EV_FULL);
        return;
    }
    for (uint32_t p = p0; p < p1; ++p) {
        const uint64_t a = halo_cut(p);
        const uint64_t b = lead ? poff[p] : a, e = lead ? a : poff[p + 1];
        for (uint64_t j = b; j < e; ++j, ++at) {
            const trig_hit h = load_hit(hits + j);
            keys[at] = ((uint64_t)(uint32_t)(h.t_ns - base) << 32) | ((uint64_t)h.pmt << 16) | h.charge;
        }
    }
    __syncthreads();
    const uint64_t dst0 = lead ? 0 : d.n_hits - total;
    for (uint32_t i = tid; i < total; i += kEvHaloThreads) {
        const uint64_t k = keys[i];
        uint32_t r = 0;
        for (uint32_t j = 0; j < total; ++j) {
            const uint64_t o = keys[j];
            r += (o < k) || (o == k && j < i);
        }
        trig_hit h;
        h.t_ns = base + (int64_t)(k >> 32);
        h.pmt = (uint16_t)(k >> 16);
        h.charge = (uint16_t)k;
        h.reserved = 0;
        d.dbg_merged[dst0 + r] = h;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kEvHaloThreads) k_evhalo(const BatchHeader *__restrict__ hdr,
                                                           const SliceDesc *__restrict__ desc)
{
    if (hdr->err) return;           // the tile pass gave up: its per-tile outputs are not valid
    extern __shared__ __align__(16) unsigned char ev_smem[];
    uint64_t *keys = reinterpret_cast<uint64_t *>(ev_smem);
    uint32_t *psum = reinterpret_cast<uint32_t *>(keys + TRIG_EV_HALO_MAX);
    for (uint32_t s = blockIdx.x; s < hdr->n_slices; s += gridDim.x) {
        const SliceDesc &d = desc[s];
        if (!d.ev || d.ev_cap == 0 || d.n_hits == 0) continue;
        if (d.stats->flags & (TRIG_FLAG_BAD_PMT | TRIG_FLAG_UNSORTED | TRIG_FLAG_OUT_OF_RANGE)) continue;
        ev_halo_side(d, true, keys, psum, d.in_lo, d.t0);
        ev_halo_side(d, false, keys, psum, d.t0 + d.slice_ns, d.t0 + d.slice_ns);
    }
}

// Offsets of the windows in the event output: exclusive prefix of their hit
// counts (one block per slice); the total is n_events.
__global__ void __launch_bounds__(1024) k_escan(const BatchHeader *__restrict__ hdr, const SliceDesc *__restrict__ desc)
{
    if (hdr->err) return;           // the tile pass gave up: its per-tile outputs are not valid
    __shared__ uint32_t wsum[33];
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5, nwp = blockDim.x >> 5;
    for (uint32_t s = blockIdx.x; s < hdr->n_slices; s += gridDim.x) {
        const SliceDesc &d = desc[s];
        if (!d.ev || d.ev_cap == 0) continue;
        if (d.stats->flags & (TRIG_FLAG_BAD_PMT | TRIG_FLAG_UNSORTED | TRIG_FLAG_OUT_OF_RANGE | TRIG_FLAG_TRIG_FULL |
                              TRIG_FLAG_WIN_FULL)) {
            if (tid == 0) d.stats->n_events = 0;
            continue;
        }
        const uint32_t nw = (uint32_t)min((unsigned long long)d.stats->n_windows, (unsigned long long)d.win_cap);
        uint32_t carry = 0;
        for (uint32_t base = 0; base < nw; base += blockDim.x) {
            const uint32_t i = base + tid;
            const uint32_t v = i < nw ? (uint32_t)d.windows[i].n_hits : 0u;
            const uint32_t incl = warp_incl_scan(v);
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                const uint32_t w = lane < nwp ? wsum[lane] : 0u;
                const uint32_t wi = warp_incl_scan(w);
                if (lane < nwp) wsum[lane] = wi - w;
                if (lane == nwp - 1) wsum[32] = wi;
            }
            __syncthreads();
            if (i < nw) d.ev_off[i] = carry + wsum[warp] + incl - v;
            carry += wsum[32];
            __syncthreads();
        }
        if (tid == 0) {
            d.ev_off[nw] = carry;
            d.stats->n_events = carry;
            if (carry > d.ev_cap) atomicOr(&d.stats->flags, TRIG_FLAG_EV_FULL);
        }
        __syncthreads();
    }
}

// The event output: event e of window w is merged hit win_rlo[w] + e -
// ev_off[w].  A warp takes kEvRun consecutive events: it finds the first
// one's window in a 32-way search, then walks the windows (hundreds of hits
// each) forward, four copies in flight per lane.  Bound by HBM (32 bytes an
// event): 45 M events take 0.23 ms (6.3 TB/s), 0.35 with a search over all
// windows for each event.
// Slices with any capacity flag (including a skipped 1 ns tile piece, whose
// rows the merged stream lacks) copy nothing.
constexpr uint32_t kEvRun = 1024;

__global__ void __launch_bounds__(256) k_events(const BatchHeader *__restrict__ hdr, const SliceDesc *__restrict__ desc)
{
    if (hdr->err) return;           // the tile pass gave up: its per-tile outputs are not valid
    const uint32_t lane = lane_id();
    const uint64_t gw = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    uint64_t taken = 0;                     // runs of the slices before, so that each warp's share goes round
    for (uint32_t s = 0; s < hdr->n_slices; ++s) {
        const SliceDesc &d = desc[s];
        if (!d.ev || d.ev_cap == 0) continue;
        if (d.stats->flags & (TRIG_FLAG_BAD_PMT | TRIG_FLAG_UNSORTED | TRIG_FLAG_OUT_OF_RANGE | TRIG_FLAG_TRIG_FULL |
                              TRIG_FLAG_WIN_FULL | TRIG_FLAG_EV_FULL | TRIG_FLAG_TILE_FULL))
            continue;
        const uint32_t nw = (uint32_t)min((unsigned long long)d.stats->n_windows, (unsigned long long)d.win_cap);
        const uint32_t ne = (uint32_t)d.stats->n_events;
        const uint64_t runs = ((uint64_t)ne + kEvRun - 1) / kEvRun;
        const uint32_t *off = d.ev_off;
        for (uint64_t run = (gw + nwarps - taken % nwarps) % nwarps; run < runs; run += nwarps) {
            const uint32_t e0 = (uint32_t)run * kEvRun, e1 = min(ne, e0 + kEvRun);
            // last w with off[w] <= e0
            uint32_t lo = 0, hi = nw;
            while (hi - lo > 1) {
                const uint32_t step = (hi - lo + 31) / 32, at = lo + (lane + 1) * step;
                const uint32_t le = __popc(__ballot_sync(0xffffffffu, at < hi && off[at] <= e0));
                lo += le * step;
                hi = min(hi, lo + step);
            }
            uint32_t w = lo, next = off[w + 1], base = d.win_rlo[w] - off[w];
            for (uint32_t x = e0; x < e1; x += 128) {
                int4 v[4];
                bool in[4];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {
                    const uint32_t e = x + u * 32 + lane;
                    in[u] = e < e1;
                    if (in[u] && e >= next) {
                        do next = off[++w + 1];
                        while (e >= next);
                        base = d.win_rlo[w] - off[w];
                    }
                    in[u] = in[u] && CHECK(18, base + e, d.n_hits) && CHECK(19, e, d.ev_cap);
                    if (in[u]) v[u] = *reinterpret_cast<const int4 *>(d.dbg_merged + (base + e));
                }
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u)
                    if (in[u]) *reinterpret_cast<int4 *>(d.ev + (x + u * 32 + lane)) = v[u];
            }
        }
        taken += runs;
    }
}

// ----------------------------------------------------------------- k_rank0

// Merged rank of each slice's first owned hit (hits before t0 are the
// leading halo); row outputs are indexed from it.
__global__ void k_rank0(const BatchHeader *__restrict__ hdr, SliceDesc *__restrict__ desc)
{
    const uint32_t s = blockIdx.x;
    if (s >= hdr->n_slices) return;
    SliceDesc &d = desc[s];
    uint64_t r = 0, r1 = 0;
    const bool offsets = d.n_hits && !(d.stats->flags & TRIG_FLAG_BAD_PMT);       // checked, and not found wrong
    for (uint32_t p = threadIdx.x; offsets && p < d.n_pmt; p += blockDim.x) {
        uint64_t sp = d.pmt_off[p], ep = d.pmt_off[p + 1];
        uint64_t a = lb_time(d.hits, sp, ep, d.t0);
        r += a - sp;
        r1 += lb_time(d.hits, a, ep, d.t0 + d.slice_ns) - sp;
    }
    r = warp_sum_u64(r);
    r1 = warp_sum_u64(r1);
    __shared__ unsigned long long acc, acc1;
    if (threadIdx.x == 0) acc = acc1 = 0;
    __syncthreads();
    if (lane_id() == 0) {
        atomicAdd(&acc, (unsigned long long)r);
        atomicAdd(&acc1, (unsigned long long)r1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        d.dbg_rank0 = acc;
        d.dbg_rank1 = acc1;
    }
}

// -------------------------------------------------------------- k_prepend

// Largest p in [0, P) with off[p] <= x, for non-decreasing offsets with
// off[0] = 0 <= x < off[P].
__device__ __forceinline__ uint32_t run_of(const uint64_t *off, uint32_t P, uint64_t x)
{
    uint32_t lo = 0, hi = P;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (off[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// A continuation submission ("Preparation in CPU": at the end of a slice the
// trigger proceeds on the first hits of the next one; here the next slice
// starts on the last hits of the previous one): PMT p's stream of the
// combined slice is the detector's resident tail of p followed by the
// submission's hits of p.  Tail hit j of PMT p lands at j + fresh_off[p],
// fresh hit i at i + tail_off[p + 1]; the combined offsets are the sums.
__global__ void k_prepend(const trig_hit *__restrict__ tail, const uint64_t *__restrict__ tail_off, uint64_t n_tail,
                          const trig_hit *__restrict__ fresh, const uint64_t *__restrict__ fresh_off,
                          uint64_t n_fresh, uint32_t P, trig_hit *__restrict__ out, uint64_t *__restrict__ out_off)
{
    const uint64_t n = n_tail + n_fresh, total = n + P + 1;
    for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (uint64_t)gridDim.x * blockDim.x) {
        if (x >= n) {
            const uint64_t q = x - n;
            out_off[q] = tail_off[q] + fresh_off[q];
            continue;
        }
        const trig_hit *src;
        uint64_t dst;
        if (x < n_tail) {
            const uint32_t p = run_of(tail_off, P, x);
            src = tail + x;
            dst = x + fresh_off[p];
        } else {
            const uint64_t i = x - n_tail;
            const uint32_t p = run_of(fresh_off, P, i);
            src = fresh + i;
            dst = i + tail_off[p + 1];
        }
        if (CHECK(21, dst, n)) *reinterpret_cast<int4 *>(out + dst) = *reinterpret_cast<const int4 *>(src);
    }
}

cudaError_t launch_prepend(const trig_hit *tail, const uint64_t *tail_off, uint64_t n_tail, const trig_hit *fresh,
                           const uint64_t *fresh_off, uint64_t n_fresh, uint32_t P, trig_hit *out, uint64_t *out_off,
                           cudaStream_t st)
{
    const uint64_t total = n_tail + n_fresh + P + 1;
    const uint64_t blocks = std::min<uint64_t>((total + 255) / 256, (uint64_t)device_sm_count() * 16);
    k_prepend<<<(unsigned)blocks, 256, 0, st>>>(tail, tail_off, n_tail, fresh, fresh_off, n_fresh, P, out, out_off);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- k_status

// The status again after event extraction, which may add TRIG_FLAG_EV_FULL.
__global__ void k_status(const BatchHeader *__restrict__ hdr, const SliceDesc *__restrict__ desc)
{
    const uint32_t n = hdr->n_slices;
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        trig_slice_stats *st = desc[s].stats;
        const uint32_t f = st->flags | hdr->err;
        st->flags = f;
        st->status = status_of(f);
    }
}

#ifdef TRIG_PHASE_STATS
// Tile-kernel counters of the phase-statistics build (summed over blocks
// since the last reset): read n of them into out, then optionally reset.
extern "C" int trig_phase_stats(unsigned long long *out, int n, int reset)
{
    unsigned long long v[24] = {};
    if (n > 24) n = 24;
    if (cudaMemcpyFromSymbol(v, g_phase, sizeof v) != cudaSuccess) return -1;
    for (int i = 0; i < n; ++i) out[i] = v[i];
    if (reset) {
        const unsigned long long z[24] = {};
        if (cudaMemcpyToSymbol(g_phase, z, sizeof z) != cudaSuccess) return -1;
    }
    return 0;
}
#endif

#ifdef TRIG_CHECK
// First recorded check failure of the process (checked builds only).
extern "C" int trig_check_record(unsigned *site, unsigned *count, unsigned long long *index,
                                 unsigned long long *limit)
{
    CheckRecord r{};
    if (cudaMemcpyFromSymbol(&r, g_check, sizeof r) != cudaSuccess) return -1;
    *site = r.site;
    *count = r.count;
    *index = r.index;
    *limit = r.limit;
    return 0;
}
#endif

// ------------------------------------------------- static scratch array

// Scratch of trig_batch_run_noalloc: a fixed device array, present on every
// device that loads the library until the process exits.  Calls share it
// and it keeps the previous call's contents; k_put clears the counters
// that must start at zero, and everything else is written before it is
// read.  Calls that overlap on the GPU race on it.
static __device__ __align__(256) unsigned char g_noalloc_scratch[TRIG_NOALLOC_SCRATCH_BYTES];

// Device address of the array for the current device, looked up once per
// device (host code may not use the symbol's name as an address).
cudaError_t static_scratch(void **ptr, size_t *bytes)
{
    static std::mutex mu;
    static void *addr[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e) return e;
        addr[dev] = p;
    }
    *ptr = addr[dev];
    *bytes = sizeof(g_noalloc_scratch);
    return cudaSuccess;
}

// ------------------------------------------------------------------- k_put

// The batch's header and descriptors (K slices of them at a time) travel as
// the kernel's parameter, copied when it is launched or captured: nothing is
// read from host memory later, no copy waits on the caller's stream, and a
// captured graph names no host or device allocation but through the kernels'
// own pointers.  The same launch zeroes the slices' counters.
template <uint32_t K>
struct PutPlan {
    BatchHeader hdr;
    uint32_t first, n;          // descriptors [first, first + n) of the batch
    SliceDesc desc[K];
};
static_assert(sizeof(BatchHeader) % 4 == 0 && sizeof(SliceDesc) % 4 == 0, "copied as 32-bit words");
static_assert(sizeof(PutPlan<kPutSlices>) <= 32000, "kernel parameter space");

template <uint32_t K>
__global__ void __launch_bounds__(256) k_put(const __grid_constant__ PutPlan<K> plan, BatchHeader *hdr, SliceDesc *desc)
{
    let_next_kernel_in();
    const uint32_t tid = threadIdx.x, at = blockIdx.x * 256 + tid;
    const uint32_t *src_h = reinterpret_cast<const uint32_t *>(&plan.hdr);
    const uint32_t *src_d = reinterpret_cast<const uint32_t *>(plan.desc);
    if (plan.first == 0 && at < sizeof(BatchHeader) / 4) reinterpret_cast<uint32_t *>(hdr)[at] = src_h[at];
    uint32_t *dst = reinterpret_cast<uint32_t *>(desc + plan.first);
    for (uint32_t i = at; i < plan.n * (uint32_t)(sizeof(SliceDesc) / 4); i += gridDim.x * 256) dst[i] = src_d[i];
    if (at < plan.n) {
        trig_slice_stats z{};
        z.n_hits = plan.desc[at].n_hits;
        *plan.desc[at].stats = z;
    }
}

template <uint32_t K>
static cudaError_t put_part(const BatchHeader &hdr, const SliceDesc *desc, uint32_t first, uint32_t n, BatchHeader *d_hdr,
                            SliceDesc *d_desc, cudaStream_t st)
{
    static_assert(sizeof(BatchHeader) / 4 <= 256, "a word per thread");
    PutPlan<K> plan;
    plan.hdr = hdr;
    plan.first = first;
    plan.n = n;
    std::memcpy(plan.desc, desc + first, n * sizeof(SliceDesc));
    // a block per two descriptors (reads of the parameter by 32 different
    // addresses take turns: 17 us for 64 of them in one block)
    k_put<K><<<(n + 1) / 2, 256, 0, st>>>(plan, d_hdr, d_desc);
    return cudaGetLastError();
}

// The parameter is as large as the smallest of four sizes that holds the
// descriptors: a launch copies it whole (30 KB at 64 slices).
static cudaError_t launch_put(const BatchHeader &hdr, const SliceDesc *desc, BatchHeader *d_hdr, SliceDesc *d_desc,
                              cudaStream_t st, uint64_t *nl)
{
    for (uint32_t first = 0; first < hdr.n_slices; first += kPutSlices) {
        const uint32_t n = std::min(kPutSlices, hdr.n_slices - first);
        cudaError_t e;
        if (n <= 1) e = put_part<1>(hdr, desc, first, n, d_hdr, d_desc, st);
        else if (n <= 4) e = put_part<4>(hdr, desc, first, n, d_hdr, d_desc, st);
        else if (n <= 16) e = put_part<16>(hdr, desc, first, n, d_hdr, d_desc, st);
        else e = put_part<kPutSlices>(hdr, desc, first, n, d_hdr, d_desc, st);
        if (e != cudaSuccess) return e;
        ++*nl;
    }
    return cudaSuccess;
}

// ------------------------------------------------------------------ launch

int device_sm_count()
{
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

// The dynamic shared memory limit of a kernel is per-function state that
// CUDA graphs do not capture: a graph replayed after the limit was lowered
// for a smaller launch would exceed it.  So each tile kernel's limit is set
// once per device, to the device's opt-in maximum, and never lowered.
template <typename K>
static cudaError_t raise_smem_limit(K kern, bool *done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (done[dev]) return cudaSuccess;
    int optin = 0;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, kern))) return e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  optin - (int)fa.sharedSizeBytes)))
        return e;
    done[dev] = true;
    return cudaSuccess;
}

template <int CAP, int NC, bool SMEM_DT, bool EXT = false, bool DENSE = false>
static cudaError_t launch_tile(BatchHeader *hdr, SliceDesc *desc, uint32_t max_pmt, cudaStream_t st)
{
    static bool limit_set[64] = {};
    size_t smem = TileLayout<CAP, NC, SMEM_DT, EXT>::bytes(max_pmt);
    auto kern = k_tile<CAP, NC, SMEM_DT, EXT, DENSE>;
    cudaError_t e = raise_smem_limit(kern, limit_set);
    if (e != cudaSuccess) return e;
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NC + 32, smem);
    if (per_sm < 1) per_sm = 1;
    return launch_next(kern, device_sm_count() * per_sm, NC + 32, smem, st, hdr, desc, max_pmt);
}

const char *const kKernelNames[kPipelineKernels] = {"k_put",   "k_bounds", "k_scatter", "k_tile",  "k_evhalo",
                                                     "k_final", "k_escan",  "k_events",  "k_status"};

cudaError_t launch_batch(const BatchHeader &hdr, const SliceDesc *desc, BatchHeader *d_hdr, SliceDesc *d_desc,
                         uint32_t max_pmt, bool any_smem_dt, const TileConfig &cfg, cudaStream_t st, uint64_t *launches,
                         bool rows, cudaEvent_t *ev)
{
    const int sms = device_sm_count();
    const uint32_t n_slices = hdr.n_slices;
    const bool any_wide = hdr.any_wide != 0, any_events = hdr.any_events != 0, any_ext = hdr.any_ext != 0;
    const bool dense = hdr.dense != 0;
    cudaError_t e;
    auto mark = [&](int i) {
        if (ev) cudaEventRecord(ev[i], st);
    };
    const uint32_t sb = n_slices < (uint32_t)sms * 4 ? n_slices : (uint32_t)sms * 4;
    uint64_t nl = 0;
    mark(0);
    if ((e = launch_put(hdr, desc, d_hdr, d_desc, st, &nl)) != cudaSuccess) return e;
    mark(1);
    if ((e = launch_next(k_bounds, sms * 6, kBoundsThreads, 0, st, d_hdr, d_desc)) != cudaSuccess) return e;
    nl += 1;
    if (rows) {
        k_rank0<<<n_slices, 256, 0, st>>>(d_hdr, d_desc);
        nl += 1;
    }
    mark(2);
    if (any_wide) {
        if ((e = launch_next(k_scatter, sms * 4, kScatThreads, 0, st, d_hdr, d_desc)) != cudaSuccess) return e;
        nl += 1;
    }
    mark(3);
    const bool smem_dt = any_smem_dt && max_pmt <= kSmemDtMaxPmt;
    if (any_ext || any_events || rows) {
        // level 0, seed rule 1, distinct count, and every batch that needs
        // the merged rows (event extraction, row outputs): the extended
        // builds, which put a tile in full (t, pmt, charge) order for the
        // rows and for level 0 over different PMTs
        if (cfg.cap == 1024)
            e = smem_dt ? launch_tile<1024, 128, true, true>(d_hdr, d_desc, max_pmt, st)
                        : launch_tile<1024, 128, false, true>(d_hdr, d_desc, max_pmt, st);
        else if (cfg.cap == 2048 && cfg.warps == 16)
            e = smem_dt ? launch_tile<2048, 512, true, true>(d_hdr, d_desc, max_pmt, st)
                        : launch_tile<2048, 512, false, true>(d_hdr, d_desc, max_pmt, st);
        else if (cfg.cap == 2048)
            e = smem_dt ? launch_tile<2048, 256, true, true>(d_hdr, d_desc, max_pmt, st)
                        : launch_tile<2048, 256, false, true>(d_hdr, d_desc, max_pmt, st);
        else if (cfg.warps == 8)
            e = smem_dt ? launch_tile<4096, 256, true, true>(d_hdr, d_desc, max_pmt, st)
                        : launch_tile<4096, 256, false, true>(d_hdr, d_desc, max_pmt, st);
        else
            e = smem_dt ? launch_tile<4096, 512, true, true>(d_hdr, d_desc, max_pmt, st)
                        : launch_tile<4096, 512, false, true>(d_hdr, d_desc, max_pmt, st);
    } else if (dense) {
        // a warp per seed in the causal count; dt rows read through the cache
        if (cfg.cap == 1024)
            e = launch_tile<1024, 128, false, false, true>(d_hdr, d_desc, max_pmt, st);
        else if (cfg.cap == 2048)
            e = cfg.warps == 16 ? launch_tile<2048, 512, false, false, true>(d_hdr, d_desc, max_pmt, st)
                                : launch_tile<2048, 256, false, false, true>(d_hdr, d_desc, max_pmt, st);
        else
            e = cfg.warps == 8 ? launch_tile<4096, 256, false, false, true>(d_hdr, d_desc, max_pmt, st)
                               : launch_tile<4096, 512, false, false, true>(d_hdr, d_desc, max_pmt, st);
    } else if (cfg.cap == 1024)
        e = smem_dt ? launch_tile<1024, 128, true>(d_hdr, d_desc, max_pmt, st)
                    : launch_tile<1024, 128, false>(d_hdr, d_desc, max_pmt, st);
    else if (cfg.cap == 2048 && cfg.warps == 16)
        e = smem_dt ? launch_tile<2048, 512, true>(d_hdr, d_desc, max_pmt, st)
                    : launch_tile<2048, 512, false>(d_hdr, d_desc, max_pmt, st);
    else if (cfg.cap == 2048)
        e = smem_dt ? launch_tile<2048, 256, true>(d_hdr, d_desc, max_pmt, st)
                    : launch_tile<2048, 256, false>(d_hdr, d_desc, max_pmt, st);
    else if (cfg.warps == 8)
        e = smem_dt ? launch_tile<4096, 256, true>(d_hdr, d_desc, max_pmt, st)
                    : launch_tile<4096, 256, false>(d_hdr, d_desc, max_pmt, st);
    else
        e = smem_dt ? launch_tile<4096, 512, true>(d_hdr, d_desc, max_pmt, st)
                    : launch_tile<4096, 512, false>(d_hdr, d_desc, max_pmt, st);
    if (e != cudaSuccess) return e;
    mark(4);
    if (any_events) {
        static bool ev_limit_set[64] = {};
        int dev = 0;
        if ((e = cudaGetDevice(&dev))) return e;
        const int ev_smem = (int)(TRIG_EV_HALO_MAX * 8 + kEvHaloThreads * 4);
        if (dev >= 0 && dev < 64 && !ev_limit_set[dev]) {
            if ((e = cudaFuncSetAttribute(k_evhalo, cudaFuncAttributeMaxDynamicSharedMemorySize, ev_smem))) return e;
            ev_limit_set[dev] = true;
        }
        k_evhalo<<<sb, kEvHaloThreads, ev_smem, st>>>(d_hdr, d_desc);
        nl += 1;
    }
    mark(5);
    // at most as many blocks as there are chunks of tiles
    if ((e = launch_next(k_final, std::min<uint32_t>(hdr.n_fin, (uint32_t)sms * 8), kFinThreads, 0, st, d_hdr, d_desc)) !=
        cudaSuccess)
        return e;
    mark(6);
    if (any_events) {
        k_escan<<<sb, 1024, 0, st>>>(d_hdr, d_desc);
        mark(7);
        k_events<<<sms * 8, 256, 0, st>>>(d_hdr, d_desc);
        mark(8);
        k_status<<<1, 256, 0, st>>>(d_hdr, d_desc);
        nl += 3;
    } else {
        mark(7);
        mark(8);
    }
    mark(9);
    nl += 2;
    if (launches) *launches += nl;
    return cudaGetLastError();
}

}  // namespace trig
