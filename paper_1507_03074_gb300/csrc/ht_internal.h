// Internal host/device interface between the C ABI (ht_api.cu) and the
// kernels (ht_kernels.cu).  Not installed; not part of the ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "ht_device.cuh"

namespace htk {

// Privatised fill: A-strip of W rows per work item (u16 counters; W/2 rows
// per pass when a slice holds >= 65536 hits and needs u32 counters).
struct FillCfg {
    uint32_t W;           // rows per item (power of two, divides threads)
    uint32_t strips;      // ceil(n_a / W)
    uint32_t pitch16;     // tile words per row in u16 mode (multiple of 32)
    uint32_t pitch32;     // tile words per row in u32 mode (multiple of 32)
    uint32_t HC;          // vote lines staged in shared memory per chunk
    uint32_t tile_words;  // W * pitch16
    uint32_t threads;     // block size
    uint32_t accumulate;  // add the tile to M_H instead of storing it
    uint32_t dyn;         // 1: the last dyn_items() items are handed out at run time (see below)
    uint32_t bulk;        // fused fill: 1 = passes leave through u32 staging and bulk copies (k_fill_bulk)
    uint32_t vote_weight; // cost of one vote against one cell written, in the static split (cta_items)
};

// The tile fill (k_fill_tma): passes of W A-rows, each voted by one warp into
// a u32 tile of its own that leaves as a bulk copy.
struct TileCfg {
    uint32_t W;           // A rows per pass (a power of two)
    uint32_t strips;      // ceil(n_a / W) passes per (event, slice)
    uint32_t tile_words;  // max(W, 2) rows of n_b words and 3 (a pass starts anywhere inside 16 bytes), a multiple of 4
    uint32_t warps;       // per CTA
    uint32_t run;         // neighbouring passes of a CTA's run (= warps)
    uint32_t threads;     // the tuning's fill_threads (at least 32 * warps)
    uint32_t vote_agg;    // warp-aggregated vote increments (match.any + one add)
    // > 0: CTAs of kTileWarps warps, which together vote the passes of crowded
    // units (team_passes): those that are more than 1 / (team_share * CTAs) of all
    uint32_t team_share;
    uint32_t edges_later; // tiles that go to M_H: comparisons across passes are left to k_edges
};
constexpr uint32_t kTileWarps = 12;    // most warps of a tile-fill CTA (two such CTAs per SM: 80 registers a thread)
// An asked-for height (fill_rows) is halved until an SM holds this many warps:
// with 3 (16 rows of 1024) a peaks-only paper event takes 39.3 us in flight, with
// 6 26.4 us, with 12 20.2 us; with 1 (32 rows) a paper event takes 121.7 us.
constexpr uint32_t kTileMinWarps = 6;
constexpr uint32_t kTileCand = 127;    // cells >= T that a pass lists (more: every cell is looked at)
constexpr uint32_t kAhead = 4;         // lines per lane loaded ahead
// Fewest hits of a unit whose passes whole CTAs may take: at 192 units of 256 hits
// lose by it (64 slices of 128 x 1024 bins, threshold 10: 53.7 us against 33.0 us).
constexpr uint32_t kTeamHits = 512;
constexpr uint32_t kListHits = 128;    // most hits of a pass that searches its list without a look at the cost
constexpr uint32_t kHandedOut = 3;     // passes per warp handed out at run time (at least)
// words of a warp's bits (one per tile cell), of its list (the length and the cells), and of all its shared memory
__host__ __device__ constexpr uint32_t tile_bit_words(uint32_t tile_words) { return (tile_words / 32u + 4u) & ~3u; }
__host__ __device__ constexpr uint32_t tile_list_words() { return (1u + kTileCand + 3u) & ~3u; }
__host__ __device__ constexpr uint32_t tile_warp_words(uint32_t tile_words)
{
    return tile_words + tile_bit_words(tile_words) + tile_list_words() + 32u;
}
inline size_t tile_smem_bytes(const TileCfg &c) { return (size_t)c.warps * tile_warp_words(c.tile_words) * 4; }
constexpr uint32_t kOrderPasses = 256; // threads of a k_order_passes or k_edges CTA, and most passes of its segment
__host__ __device__ inline uint64_t tile_passes(const Geom &g, const TileCfg &c, uint32_t n_events)
{
    return (uint64_t)n_events * g.n_slices * c.strips;
}

// Shared-memory words of the fused fill's two u32 staging buffers (half a
// u16 pass, W / 2 rows of n_b cells, each), or 0 without bulk copies.
__host__ __device__ constexpr uint32_t staging_words(const FillCfg &c, uint32_t nb) { return c.bulk ? c.W * nb : 0u; }

// The fills split the first items - dyn_items(items, grid) work items over
// their CTAs by estimated cost, and hand the rest out one at a time to the
// CTAs that finish first (an atomic counter), which absorbs the spread of
// the static split.  In the fused fill every handed-out item gets its own
// list of candidate chunks, numbered grid + its rank, so the lists stay in
// linear order.
__host__ __device__ constexpr uint64_t dyn_items(uint64_t items, uint32_t grid)
{
    return items / 8 < 2ull * grid ? items / 8 : 2ull * grid;
}

// Scan (and its chunk bookkeeping).  Shared with k_order.
struct ScanArgs {
    uint32_t grid;        // persistent CTAs (each owns a contiguous run of rows)
    uint32_t R;           // own rows per stage (bulk) / per chunk (streaming, direct)
    uint32_t S;           // stages in the shared-memory ring (<= 8)
    uint32_t K;           // peak entries buffered in shared memory (>= 2*256)
    uint32_t slot_words;  // (R + 2) * n_b
    uint32_t hot_words;   // streaming: words of the per-CTA hot-chunk bitmap
    uint32_t seq_max;     // chunk descriptors per CTA
    uint32_t entries_cap; // global entry scratch capacity
    uint4 *entries;       // {lin within event, event, votes, 0}
    uint32_t *g_count;    // entries used (reset by k_order)
    uint2 *desc;          // [grid][seq_max] {base, n}
    uint32_t *cta_nseq;   // [grid] interior chunks
    uint32_t *cta_total;  // [grid] entries
    uint32_t *ev_count;   // [n_events] peaks per event (reset by k_order)
};

struct OrderArgs {
    Peak *out;            // [n_events][capacity]
    uint32_t capacity;
    uint32_t *counts;     // [n_events] total peaks per event
    uint32_t *ev_count;
    uint32_t *ticket;     // last-CTA detection (reset by k_order)
    uint32_t *g_count;    // entries used (reset by the last CTA)
    uint32_t compact;     // 1: one list out[rank] over all events, else out[e][capacity]
    uint32_t *status_out; // receives the status word (mapped host memory), or nullptr
};

cudaError_t launch_bin(const Geom &g, const Work &w, uint32_t grid, cudaStream_t st);
cudaError_t launch_scatter(const Geom &g, const Work &w, uint32_t grid, cudaStream_t st);
// k_bin + k_scatter as one cluster of cs <= kBinClusterMax CTAs of
// kBinClusterThreads threads, each holding at most kBinClusterHPT hits: for
// launches of at most kBinClusterMax * kBinClusterThreads * kBinClusterHPT hits
// whose three words per unit and hit offsets fit kBinClusterSmem bytes.
// 512 threads of 64 registers and 10 KB of shared memory fit on an SM beside two
// CTAs of the tile fill, so an event's binning runs under the fill of the event
// before it (three contexts in flight, against CTAs of 1024 threads: paper event
// 37.3 -> 33.8 us, peaks only 23.4 -> 20.0 us; one context alone 35.6 against
// 34.5 us, peaks only).
constexpr uint32_t kBinClusterMax = 8, kBinClusterThreads = 512, kBinClusterHPT = 4;
constexpr size_t kBinClusterSmem = 40 * 1024;
size_t bin_cluster_smem_bytes(const Geom &g, uint32_t n_events);
cudaError_t launch_bin_cluster(const Geom &g, const Work &w, uint32_t cs, cudaStream_t st);
// Whether this device runs a cluster of kBinClusterMax such CTAs.
bool bin_cluster_supported(size_t smem);
size_t fill_smem_bytes(const FillCfg &c);
cudaError_t launch_fill_priv(const Geom &g, const Work &w, const FillCfg &c, uint32_t grid,
                             cudaStream_t st);
size_t fill_scan_smem_bytes(const FillCfg &c, const ScanArgs &a, uint32_t nb);
cudaError_t launch_fill_scan(const Geom &g, const Work &w, const FillCfg &c, const ScanArgs &a, uint32_t grid,
                             cudaStream_t st);
cudaError_t fill_scan_occupancy(const FillCfg &c, const ScanArgs &a, uint32_t nb, int *blocks_per_sm);
// Warp-specialised fused fill: kWsThreads threads, two tiles (c.threads is
// the vote group's size, kWsThreads / 2).
constexpr uint32_t kWsThreads = 1024;
size_t fill_ws_smem_bytes(const FillCfg &c, const ScanArgs &a);
cudaError_t launch_fill_ws(const Geom &g, const Work &w, const FillCfg &c, const ScanArgs &a, uint32_t grid,
                           cudaStream_t st);
cudaError_t fill_ws_occupancy(const FillCfg &c, const ScanArgs &a, int *blocks_per_sm);
// The tile fill (store: M_H is written, else only the peaks are found), and the
// ordering of the peaks it leaves pass by pass (one event, or o.compact).
cudaError_t launch_fill_tma(const Geom &g, const Work &w, const TileCfg &c, const ScanArgs &a, uint32_t grid,
                            bool store, cudaStream_t st);
cudaError_t fill_tma_occupancy(const TileCfg &c, bool store, int *blocks_per_sm);
cudaError_t launch_order_passes(const Geom &g, const Work &w, const ScanArgs &a, const OrderArgs &o, uint64_t passes,
                                cudaStream_t st);
// After a tile fill with edges_later: drop its candidates that a row of another pass outdoes.
cudaError_t launch_edges(const Geom &g, const Work &w, const TileCfg &c, const ScanArgs &a, uint64_t passes,
                         cudaStream_t st);
// k_edges from this many admissions per (event, slice) on, on average.  Voting
// the rows beyond costs more the more hits a slice has, k_edges one more launch:
// paper matrix, 78 hits per slice, without and with: 33.8 and 34.0 us in flight,
// 48.7 and 51.2 us alone; 156: 36.7 and 35.9, 60.1 and 56.7; 250: 49.3 and 42.6,
// 85.2 and 69.7; windows with 169 (at most): 33.9 and 34.1, 49.2 and 53.0.
constexpr uint32_t kEdgeHits = 192;
// After k_fill_scan, k_fill_bulk or k_fill_ws (same grid): test its candidate
// entries, keep the peaks.
cudaError_t launch_peaks(const Geom &g, const Work &w, const ScanArgs &a, uint32_t grid, cudaStream_t st);
// Accumulating fills of few hits: M_H += their votes, one reduction each (kAddRows A rows of a slice per warp).
constexpr uint32_t kAddRows = 32;
cudaError_t launch_fill_add(const Geom &g, const Work &w, uint32_t num_sms, cudaStream_t st);
// n cells of M_H to device memory (both 32-byte aligned).
cudaError_t launch_copy(uint32_t *dst, const uint32_t *src, uint64_t n, cudaStream_t st);
cudaError_t launch_clear(uint32_t *M, uint64_t words, uint32_t grid, cudaStream_t st);
cudaError_t launch_fill_naive(const Geom &g, const Work &w, uint32_t num_sms, cudaStream_t st);
size_t scan_smem_bytes(const ScanArgs &a);

// Layout of the counter block: [0] status, [1] entries used, [2] order
// ticket, [3] binning ticket (reset by k_bin's last block), [4] next
// handed-out fill item and [5] fill CTAs done with them (both reset by the
// last such CTA), [6 ..) peaks per event.  k_bin zeroes words 1, 2 and
// [6, 6 + n_events) before every fill.
enum : uint32_t {
    CTR_STATUS = 0, CTR_ENTRIES = 1, CTR_OTICKET = 2, CTR_BTICKET = 3, CTR_DYN = 4, CTR_DYN_DONE = 5,
    CTR_P4TICKET = 6, CTR_TEAM = 7, CTR_EVENTS = 8
};

// Cost model of the balanced split of (event, slice, strip) work items over
// the CTAs of the fills other than the tile fill: a strip of r rows in a slice
// of h hits costs r * (n_b + v * h) (writing a cell ~ 1, one vote ~ v).
constexpr uint32_t kVoteWeight = 6;

// Scan variants: bulk-copy (TMA) ring, register streaming, direct (any n_b).
// The streaming variant keeps kLdgUPT 16-byte loads per thread in flight.
constexpr uint32_t kLdgUPT = 8;
// Candidate cells (>= threshold) a streaming-scan CTA lists before testing them.
constexpr uint32_t kCand = 1024;
// Candidate cells a fused-fill CTA lists per pass; a pass with more emits
// its rows' cells >= T read back from M_H.
constexpr uint32_t kFusedCand = 256;
// Entries the fused fill emits per group round: at most this many per
// round, so every chunk but the last holds at least K - fused_round(threads, K).
__host__ __device__ constexpr uint32_t fused_round(uint32_t threads, uint32_t K) { return threads < K / 2 ? threads : K / 2; }
enum ScanKind { SCAN_DIRECT = 0, SCAN_BULK = 1, SCAN_LDG = 2 };
cudaError_t launch_scan(const Geom &g, const Work &w, const ScanArgs &a, int kind, cudaStream_t st);
cudaError_t launch_order(const Geom &g, const Work &w, const ScanArgs &a, const OrderArgs &o,
                         cudaStream_t st);
// L2 atomic increments at pseudo-random words of buf (mask + 1 words,
// per_thread per thread, 256 threads per CTA).
cudaError_t launch_atomic_rate(uint32_t *buf, uint32_t mask, uint32_t per_thread, uint32_t seed, uint32_t grid,
                               cudaStream_t st);
// One bounded wait that nothing ends (k_wait_probe): flags ST_WAIT_TIMEOUT
// after limit_ms (at most about a second).
cudaError_t launch_wait_probe(uint32_t *status, uint32_t limit_ms, cudaStream_t st);
// The 4-D filter of a 2-D peak list (k_peaks4d): keep holds cap_in flags;
// ticket is a zero counter word (reset by the kernel).
cudaError_t launch_peaks4d(const Geom &g, const uint32_t *M, const Peak *in, const uint32_t *n_in, uint32_t cap_in,
                           uint8_t *keep, Peak *out, uint32_t cap_out, uint32_t *n_out, uint32_t *ticket,
                           uint32_t *status, uint32_t grid, cudaStream_t st);
cudaError_t scan_occupancy(int kind, size_t smem, int *blocks_per_sm);
cudaError_t fill_occupancy(const FillCfg &c, int *blocks_per_sm);

} // namespace htk
