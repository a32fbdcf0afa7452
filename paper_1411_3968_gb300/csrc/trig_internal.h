// trig_internal.h -- structures shared by the sm_103a kernels (trig_kernels.cu)
// and the host runtime (trig_engine.cpp).  Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "trig.h"

namespace trig {

// Limits of this implementation.
constexpr uint32_t kMaxPmt = 4096;          // PMTs per detector
constexpr uint32_t kSmemDtMaxPmt = 96;      // dt table lives in shared memory up to this P
constexpr uint32_t kDtRow = 256;            // bytes of a dt row in shared memory (128 PMTs)
constexpr uint32_t kWideMinPmt = 129;       // from this P on, slices are staged from a bucketed copy
constexpr uint32_t kSegBuckets = 4096;      // buckets of a segment at most (k_scatter)
// A tile plus its halos spans less than 2^20 ns, so a hit's time within the
// staged range and its PMT (< 2^12) pack into 32 bits.  The limit keeps
// 65536 ns (more than any dt, <= 60000 ns) between the last staged time and
// 2^20 - 1, the time of the end keys that the causal count may read past
// the last key.
constexpr uint32_t kTileSpanBits = 20;
constexpr int64_t kMaxTileSpan = ((int64_t)1 << kTileSpanBits) - 65536;
constexpr uint64_t kMaxSliceHits = 0xFFFFFFF0ull;

// Detector tables resident on the device (owned by trig_detector).
struct DetDev {
    uint16_t *dt;         // [P*P] min(dt_max, W), row p_s
    int32_t *dt_exact;    // [P*P] exact dt_max
    uint16_t *floor;      // [P] dense floor index
    uint16_t *dmax_row;   // [P] max_q min(dt_max[p][q], W)
    uint8_t *rel;         // [P*P] relation of PMTs p, q (seed rule 1 only), kRel* bits
};

// PMT relations of the coincidence seed rule.
constexpr uint8_t kRelFloor = 1;        // another PMT of the same floor (FC)
constexpr uint8_t kRelAdjacent = 2;     // adjacent PMT: same floor, within sc_dist (SC)
constexpr uint8_t kRelNextFloor = 4;    // PMT on a consecutive floor of the same tower (AFC)
// In shared memory the relation sits above the dt entry, which then has
// kRelShift bits (corr_window_ns below 2^13; the workloads' is 3000).
constexpr uint32_t kRelShift = 13;

// Per-slice descriptor in device scratch, written by the host each run.
struct SliceDesc {
    const trig_hit *hits;
    const uint64_t *pmt_off;
    const uint16_t *dt;
    const uint16_t *floor;
    const uint16_t *dmax_row;
    uint32_t n_pmt;
    uint32_t halo;          // tile halo H = max(max dmax_row, floor_tau)
    uint32_t q_seed;
    uint32_t tau;
    uint32_t threshold;
    uint32_t win_half;
    uint32_t l0_hits;       // level 0: N hits (0 = off) within l0_window ns,
    uint32_t l0_window;     //   of different PMTs if l0_distinct
    uint32_t l0_distinct;
    uint32_t seed_rule;     // 0: charge or floor coincidence; 1: [SC and AFC] or [FC and AFC]
    uint32_t sc_w, fc_w, afc_w;     // coincidence windows of seed rule 1 (ns)
    uint32_t count_distinct;        // c(s) counts different PMTs (P <= 128)
    const uint8_t *rel;     // [P*P] kRel* bits (seed rule 1)
    uint32_t rel_in_dt;     // seed rule 1 and every dt below 2^kRelShift
    int64_t t0;
    int64_t slice_ns;
    int64_t in_lo, in_hi;   // accepted hit times [in_lo, in_hi)
    uint64_t n_hits;
    int64_t tile_w;         // tile width W (ns); tile g owns [t0 + g W, t0 + (g+1) W)
    uint32_t w_magic;       // ceil(2^32 / edge_w): 32-bit quotient estimate when span32
    uint32_t span32;        // all in-range times are < 2^31 ns past the first edge
    uint32_t n_tiles;       // NG (<= 2^20)
    uint32_t item0;         // first work item (tile) of this slice
    uint32_t chunk0;        // first structure-pass chunk of this slice
    uint32_t *edge;         // [n_edges][P] first hit index at or past each tile edge (narrow slices):
                            //   edge 2g is B_g - H, edge 2 (g + edge_a) + 1 is B_{g+1} + H
    uint32_t n_edges, edge_a, edge_b;       // 2H + W = edge_a W + edge_b
    int64_t edge_org;       // time of the first edge
    uint32_t edge_w;        // W; wide slices: the length of a segment of seg_bkt buckets, whose
    uint32_t seg_bkt;       //   starts are their edges
    // Wide slices (P >= kWideMinPmt): the hits are also copied, grouped by
    // time bucket [O + b Wb, O + (b+1) Wb), into tbuf; tile g's core is the
    // buckets [lead + g m, lead + (g+1) m) and it stages those plus `hh`
    // buckets on each side, one contiguous range of tbuf.
    uint32_t wide;
    uint32_t bkt_w;         // Wb (ns)
    uint32_t bkt_magic;     // ceil(2^32 / Wb)
    uint32_t bkt_lead;      // buckets before t0
    uint32_t bkt_per_tile;  // m
    uint32_t bkt_halo;      // hh = ceil(H / Wb)
    uint32_t n_bkt;         // NB
    uint32_t bkt32;         // every in-range time is < 2^31 ns past O
    int64_t bkt_origin;     // O = t0 - lead * Wb
    uint32_t *bkt_off;      // [NB + 1] merged rank of each bucket's first hit
    trig_hit *tbuf;         // [n_hits] hits in bucket order
    trig_trigger *stage;    // [n_hits] fired seeds at their merged rank
    uint32_t *wrank;        // [n_hits][2] beside each staged fired seed: the merged ranks of the
                            //   first hit at or after t - win_half and of the first after t + win_half
    uint32_t *tile_nfired;  // [NG]
    uint32_t *tile_rank;    // [NG] merged rank of the tile's first core hit
    unsigned char *fin;     // this slice's chunks of tiles (FinState each), of the batch's
    uint32_t fin0;          // first of them in the batch
    trig_trigger *triggers;
    uint64_t trig_cap;
    trig_window *windows;
    uint64_t win_cap;
    trig_slice_stats *stats;
    // event extraction (ev != nullptr): the slice's hits in merged order,
    // each window's first merged rank and its offset in the event output
    trig_hit *ev;
    uint64_t ev_cap;
    uint32_t *win_rlo;      // [win_cap]
    uint32_t *ev_off;       // [win_cap + 1]
    trig_hit *dbg_merged;   // merged rows, indexed by merged rank - dbg_rank0 (row outputs,
                            // or the slice's merged stream for event extraction)
    uint32_t *dbg_seedcnt;
    uint64_t dbg_rank0;     // merged rank of the first owned hit (row outputs only)
    uint64_t dbg_rank1;     // merged rank of the first hit after the owned range
};

struct BatchHeader {
    uint32_t n_slices;
    uint32_t n_items;       // total tiles
    uint32_t n_chunks;      // total structure-pass chunks
    uint32_t err;
    uint32_t queue;         // tile work queue head
    uint32_t any_wide;      // a slice of the batch is wide
    uint32_t any_events;    // a slice of the batch extracts events
    uint32_t any_ext;       // a slice uses level 0, seed rule 1 or the distinct count
    uint32_t dense;         // a slice expects kDenseKeys or more keys per causal scan range
    uint32_t stall;         // test control: the tile pass's stagers fill nothing, so its waits run out
    uint32_t n_fin;         // chunks of kFinTiles tiles, at least one for each slice
    uint32_t fin_queue;     // next of them
    unsigned char *fin;     // their states
    uint64_t wait_ns;       // limit of every device wait (ns); a wait that runs out sets TRIG_FLAG_TIMEOUT
};

constexpr uint64_t kDefaultWaitNs = 1000000000ull;     // one second

// Expected keys in a seed's scan range (2H + 1 ns at the slice's mean rate)
// from which the causal count gives each seed a warp instead of 4 lanes.
constexpr double kDenseKeys = 600.0;

constexpr uint32_t kFinTiles = 32;          // tiles whose seeds a block of k_final takes at a time
constexpr uint32_t kFinStateBytes = 104;    // what such a chunk publishes
constexpr uint32_t kPutSlices = 64;         // descriptors a launch of k_put carries at most

constexpr uint32_t kChunkHits = 992;        // structure-pass chunk: 8 warps of 4 x 31 hits

// Kernel launch helpers implemented in trig_kernels.cu.
cudaError_t launch_dtmax(const int32_t *xyz, uint32_t n_pmt, uint32_t tol, uint32_t n_num, uint32_t n_den,
                         uint32_t corr, int32_t *dt_exact, uint16_t *dt, uint16_t *dmax_row, cudaStream_t st);

// Launch shape of the tile kernel: hits per shared-memory tile, consumer
// warps per block, and the target fill of a tile (percent of cap) that sets
// the tile width.  Valid (cap, warps): (4096, 16), (4096, 8), (2048, 16),
// (2048, 8), (1024, 4); smaller tiles run more blocks per SM (up to 2 for
// 2048 hits, 4 or more for 1024).
struct TileConfig {
    uint32_t cap;
    uint32_t warps;
    uint32_t fill_pct;
    uint32_t spread = 0;    // tiles cut smaller so that a small batch fills the GPU (kOwnShape)
    uint32_t lean = 0;      // smaller side tables (1), the smallest (2): a batch at the edge of a fixed scratch
};
// The library's own choice: the shape the autotuner ends at for towers, with
// two blocks on an SM (4096-hit tiles leave room for one: 15.7 against 20.3 us
// for 320 k hits, 72 against 83 us for 2.8 M, 1.33 against 1.68 ms for 52 M
// under the distinct count); for dense arrays it is kOwnDenseShape.
constexpr TileConfig kOwnShape{2048, 16, 90, 1};
// Many tiles of an array so dense that halos crowd the tile (see halo_heavy).
constexpr TileConfig kOwnDenseShape{4096, 16, 90, 0};
inline bool valid_tile_shape(uint32_t cap, uint32_t warps)
{
    return ((cap == 4096 || cap == 2048) && (warps == 16 || warps == 8)) || (cap == 1024 && warps == 4);
}
constexpr uint32_t kMaxTilesPerSlice = 1u << 20;

constexpr int kPipelineKernels = 9;
extern const char *const kKernelNames[kPipelineKernels];

// Enqueues the batch pipeline, the copy of its header and descriptors to
// d_hdr and d_desc included.  hdr.any_wide: the scatter kernel runs only
// then; any_events: the halo, event-offset, event-copy and
// status kernels run only then; any_ext: the tile kernel built with level 0,
// seed rule 1 and the distinct count runs, else the one without them; dense:
// the tile kernel built with a warp per seed in the causal count runs.  ev
// (optional, kPipelineKernels + 1 events): ev[i] is recorded before pipeline
// kernel i and ev[kPipelineKernels] after the last one (a kernel that does
// not run gets an empty interval).  *launches is increased by the number of
// kernels launched.
cudaError_t launch_batch(const BatchHeader &hdr, const SliceDesc *desc, BatchHeader *d_hdr, SliceDesc *d_desc,
                         uint32_t max_pmt, bool any_smem_dt, const TileConfig &cfg, cudaStream_t st, uint64_t *launches,
                         bool rows, cudaEvent_t *ev = nullptr);

int device_sm_count();

#ifdef __CUDACC__
// The pipeline's kernels are launched as programmatic dependents: one may
// start while its predecessor runs, sets up what needs no input, and waits
// here until every kernel before it has ended and its writes are visible.
// Every block of such a kernel waits, so a kernel's end implies that of all
// before it.
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel's blocks come in as soon as all of this one's have
// started.
__device__ __forceinline__ void let_next_kernel_in() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launches a kernel of the pipeline as a programmatic dependent of the one
// before it on the stream (wait_for_previous_kernel).
template <typename... P, typename... A>
inline cudaError_t launch_next(void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

#endif


// Continuation submissions: the combined slice (resident tail of each PMT,
// then the submission's hits of that PMT) into out / out_off.
cudaError_t launch_prepend(const trig_hit *tail, const uint64_t *tail_off, uint64_t n_tail, const trig_hit *fresh,
                           const uint64_t *fresh_off, uint64_t n_fresh, uint32_t P, trig_hit *out, uint64_t *out_off,
                           cudaStream_t st);

// What other translation units of the library read of a detector.
struct DetInfo {
    uint32_t n_pmt;
    const int32_t *xyz;     // host, 3 * n_pmt (the detector's copy)
    trig_params par;
    int64_t in_halo;        // accepted halo around a slice
    int device;
};
bool detector_info(const trig_detector *d, DetInfo *out);

// The library's error reporting (trig_last_error) and launch counter.
int report_error(int code, const char *msg);
int report_cuda_error(cudaError_t e, const char *what);
void count_launches(uint64_t n);

// Address and size of the library's static scratch array on the current device.
cudaError_t static_scratch(void **ptr, size_t *bytes);

}  // namespace trig
