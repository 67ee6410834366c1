// Hough-Transform kernels for sm_103a (GB300).
//
//   k_bin         one thread per hit (all events of a launch): the bin code
//                 of the hit's own (theta, phi) slice, found from FP32
//                 pseudo-angles and the edge tables (Sec. 2: the angles
//                 select the slice a hit votes in), and the per-hit terms
//                 x, x^2 + y^2, 2y of the vote.
//   k_scatter     the admitted hits into per-(event, slice) unit lists.
//   k_bin_cluster k_bin + k_scatter in one thread-block cluster for launches
//                 of few hits (distributed shared memory for the counts).
//   k_fill_tma    Step 1 fused with step 2 (default): a warp votes a pass of W
//                 A-rows into a u32 shared-memory tile of its own, laid out as
//                 M_H's rows, which leaves as one bulk copy; a vote taking a
//                 cell to T lists it, and the warp tests the listed cells in
//                 its tile.  Units of many hits are left to whole CTAs
//                 (team_passes).  k_order_passes puts the peaks in order.
//   k_edges       Crowded tile fills: peaks against the rows of other passes.
//   k_fill_add    Accumulating fills of few hits: a reduction per vote.
//   k_copy        M_H into the caller's device memory.
//   k_fill_priv   Step 1 (Sec. 2), privatised.  Work item = (event, slice,
//                 strip of W A-rows); each CTA takes a contiguous range of
//                 items.  It selects the event's hits admitted to the slice
//                 (ballot compaction into shared memory, cached while the
//                 CTA stays on that slice), votes them into a shared-memory
//                 u16 (or u32) tile with shared-memory atomics, and writes
//                 the tile to HBM once with 16-byte stores that also zero it.
//                 Every cell is written, so M_H needs no separate clear.
//   k_clear,      Step 1 as the paper's CUDA design (Sec. 3): an explicit
//   k_fill_naive  clear, then a 1-D grid over hits, a thread block over A,
//                 and one global atomicAdd per vote.
//   k_scan_tma    Step 2 (Sec. 2, Sec. 3): threshold + local maxima.  Each
//                 persistent CTA streams a contiguous run of M_H rows through
//                 a ring of shared-memory stages filled by 1-D bulk copies
//                 (TMA, mbarrier-completed).  A stage with no cell >= T (the
//                 common case) costs one 16-byte load per thread and row and
//                 one block vote; only stages holding candidates check the 8
//                 (A,B) neighbours and compact peaks, in order, into per-CTA
//                 chunks.  k_scan_direct is the same without staging, for
//                 n_b not a multiple of 4.
//   k_order       places every list's chunks at their global rank: ascending
//                 linear index per event, expanded to 32-byte peak records.
#include "ht_device.cuh"
#include "ht_internal.h"

#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <utility>

namespace htk {

// ---------------------------------------------------------------------------
// Block-wide helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v)
{
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o)
            v += n;
    }
    return v;
}

// Thread groups that share the block-level helpers below: the whole block
// (barrier 0), or a warp-aligned range of FIRST .. FIRST + N - 1 threads
// synchronising on named barrier ID (the warp-specialised fill runs two
// such groups side by side, each with its own barrier).
struct BlockGroup {
    static __device__ __forceinline__ uint32_t rank() { return threadIdx.x; }
    static __device__ __forceinline__ uint32_t size() { return blockDim.x; }
    static __device__ __forceinline__ void sync() { __syncthreads(); }
    static __device__ __forceinline__ int sync_or(int p) { return __syncthreads_or(p); }
};

template <uint32_t ID, uint32_t FIRST, uint32_t N>
struct WarpGroup {
    static_assert(FIRST % 32 == 0 && N % 32 == 0 && ID >= 1 && ID < 16, "warp-aligned group, named barrier 1..15");
    static __device__ __forceinline__ uint32_t rank() { return threadIdx.x - FIRST; }
    static __device__ __forceinline__ uint32_t size() { return N; }
    static __device__ __forceinline__ void sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }
    static __device__ __forceinline__ int sync_or(int p)
    {
        uint32_t r;
        asm volatile("{\n\t.reg .pred pi, po;\n\t"
                     "setp.ne.u32 pi, %1, 0;\n\t"
                     "bar.red.or.pred po, %2, %3, pi;\n\t"
                     "selp.u32 %0, 1, 0, po;\n\t}"
                     : "=r"(r)
                     : "r"((uint32_t)p), "n"(ID), "n"(N)
                     : "memory");
        return (int)r;
    }
};

// Programmatic dependent launch: every kernel here is launched so that it may
// start while the previous kernel of its stream finishes; it runs only
// set-up that touches no global data of earlier kernels before this wait
// (a no-op when the launch had no such dependency).
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream launch once every CTA of this one has
// passed this point (its grid_dep_wait still waits for this kernel to end).
// k_scatter and k_bin_cluster use it: the fill's set-up (clearing its tiles)
// then overlaps the binning's end.
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Exclusive scan of n values in shared memory (in place); returns the total.
// All threads of the block must call it.  wsum: >= 33 words of scratch.
__device__ uint32_t block_exclusive_scan(uint32_t *a, uint32_t n, uint32_t *wsum)
{
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    const uint32_t per = (n + bd - 1) / bd;
    const uint32_t b0 = min(tid * per, n), b1 = min(b0 + per, n);
    uint32_t s = 0;
    for (uint32_t i = b0; i < b1; ++i)
        s += a[i];
    const uint32_t incl = warp_incl_scan(s);
    const uint32_t warp = tid >> 5, lane = tid & 31u, nw = (bd + 31) >> 5;
    if (lane == 31u)
        wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t v = lane < nw ? wsum[lane] : 0u;
        const uint32_t vi = warp_incl_scan(v);
        wsum[lane] = vi - v;
        if (lane == 31u)
            wsum[32] = vi;
    }
    __syncthreads();
    uint32_t run = wsum[warp] + incl - s;
    for (uint32_t i = b0; i < b1; ++i) {
        const uint32_t v = a[i];
        a[i] = run;
        run += v;
    }
    const uint32_t total = wsum[32];
    __syncthreads();
    return total;
}

// ---------------------------------------------------------------------------
// k_bin: one thread per hit.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_bin(Geom g, Work w)
{
    __shared__ float et[1025], ep[1025];
    __shared__ uint32_t s_last, s_wsum[40];
    extern __shared__ uint32_t s_off[];   // n_events + 1 hit offsets (batches)
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    for (uint32_t i = tid; i <= g.nt; i += bd)
        et[i] = g.et[i];
    for (uint32_t i = tid; i <= g.np; i += bd)
        ep[i] = g.ep[i];
    grid_dep_wait();   // counters and hits of earlier kernels
    if (blockIdx.x == 0) {   // fresh counters for the fill and scan that follow
        if (tid == 0)
            w.ctr[CTR_ENTRIES] = w.ctr[CTR_OTICKET] = 0u;
        for (uint32_t i = tid; i < w.n_events; i += bd)
            w.ctr[CTR_EVENTS + i] = 0u;
    }
    for (uint32_t i = blockIdx.x * bd + tid; i < w.n_seg; i += gridDim.x * bd)
        w.seg_peaks[i] = 0u;
    if (w.hit_off)
        for (uint32_t i = tid; i <= w.n_events; i += bd)
            s_off[i] = w.hit_off[i];
    __syncthreads();
    const uint32_t n = w.hit_off ? min(s_off[w.n_events], w.n_hits0) : w.n_hits0;
    for (uint32_t h = blockIdx.x * bd + tid; h < n; h += gridDim.x * bd) {
        const float x = w.x[h], y = w.y[h];
        float r2;
        const uint32_t code = bin_code(g, et, ep, x, y, w.z[h], r2);
        uint32_t e = 0;
        if (w.hit_off) {   // the last event whose first hit is <= h
            uint32_t lo = 0, hi = w.n_events - 1;
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (s_off[mid] <= h)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            e = lo;
        }
        w.hits4[h] = make_float4(x, r2, __fmul_rn(2.0f, y), __uint_as_float(e));
        w.codes[h] = code;
        for_each_slice(g, code, [&](uint32_t s) { atomicAdd(&w.slice_cnt[e * g.n_slices + s], 1u); });
    }
    // the last block to finish turns the counts into unit offsets
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&w.ctr[CTR_BTICKET], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last)
        return;
    __threadfence();
    const uint32_t U = w.n_events * g.n_slices;
    constexpr uint32_t PER = 8;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < U; base += PER * bd) {
        uint32_t v[PER], sum = 0;
#pragma unroll
        for (uint32_t q = 0; q < PER; ++q) {
            const uint32_t u = base + tid * PER + q;
            v[q] = u < U ? __ldcg(&w.slice_cnt[u]) : 0u;
            sum += v[q];
        }
        const uint32_t incl = warp_incl_scan(sum);
        const uint32_t warp = tid >> 5, lane = tid & 31u, nw = (bd + 31) >> 5;
        if (lane == 31u)
            s_wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const uint32_t t = lane < nw ? s_wsum[lane] : 0u;
            const uint32_t ti = warp_incl_scan(t);
            s_wsum[lane] = ti - t;
            if (lane == 31u)
                s_wsum[32] = ti;
        }
        __syncthreads();
        uint32_t run = carry + s_wsum[warp] + incl - sum;
#pragma unroll
        for (uint32_t q = 0; q < PER; ++q) {
            const uint32_t u = base + tid * PER + q;
            if (u < U) {
                w.slice_off[u] = run;
                w.slice_fill[u] = 0u;
            }
            run += v[q];
        }
        carry += s_wsum[32];
        __syncthreads();
    }
    if (tid == 0) {
        w.slice_off[U] = carry;
        w.ctr[CTR_BTICKET] = 0u;
    }
}

// Hits into their units' lists (after k_bin), then clear the unit counts
// for the next binning.
__global__ void __launch_bounds__(256) k_scatter(Geom g, Work w)
{
    grid_dep_wait();
    grid_dep_launch();   // k_bin is complete: the fill may start its set-up
    const uint32_t n = w.hit_off ? min(__ldg(&w.hit_off[w.n_events]), w.n_hits0) : w.n_hits0;
    const uint32_t stride = gridDim.x * blockDim.x, t0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (uint32_t h = t0; h < n; h += stride) {
        const uint32_t code = w.codes[h];
        if (code == kDropped)
            continue;
        const float4 hv = w.hits4[h];
        const float2 line = vote_line(g, hv.x, hv.y, hv.z);
        const uint32_t e = __float_as_uint(hv.w);
        for_each_slice(g, code, [&](uint32_t s) {
            const uint32_t u = e * g.n_slices + s;
            const uint32_t idx = w.slice_off[u] + atomicAdd(&w.slice_fill[u], 1u);
            if (idx < w.list_cap) {
                w.list[idx] = hv;
                w.lines[idx] = line;
            }
        });
    }
    const uint32_t U = w.n_events * g.n_slices;
    for (uint32_t u = t0; u < U; u += stride)
        w.slice_cnt[u] = 0u;
}

// k_bin and k_scatter in one launch for launches of few hits: one cluster of
// up to kBinClusterMax CTAs.  Each CTA counts its hits per unit in its own
// shared memory; after one cluster barrier every CTA reads all the CTAs'
// counts (distributed shared memory) and derives by itself the unit totals,
// its own place inside every unit (the counts of the CTAs ranked below it)
// and, by an exclusive scan of the totals, the unit offsets.  It then lists
// its hits with local cursors.  No CTA writes another's shared memory, and
// the only other cluster barrier (split into arrive and wait) keeps every
// CTA's counts alive until all have read them.  Each thread keeps its (at
// most kBinClusterHPT) hits in registers between counting and listing.
// Dynamic shared memory: U counts, U + 1 totals / offsets, U places and
// n_events + 1 hit offsets, where U = n_events * n_slices.
__global__ void __launch_bounds__(kBinClusterThreads, 2) k_bin_cluster(Geom g, Work w)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ float et[1025], ep[1025];
    __shared__ uint32_t s_wsum[40];
    extern __shared__ uint32_t s_cnt[];
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    const uint32_t rank = cl.block_rank(), cs = cl.num_blocks();
    const uint32_t U = w.n_events * g.n_slices;
    uint32_t *s_tot = s_cnt + U, *s_pl = s_tot + U + 1, *s_off = s_pl + U;
    for (uint32_t i = tid; i <= g.nt; i += bd)
        et[i] = g.et[i];
    for (uint32_t i = tid; i <= g.np; i += bd)
        ep[i] = g.ep[i];
    for (uint32_t u = tid; u < U; u += bd)
        s_cnt[u] = 0u;
    grid_dep_wait();     // counters and hits of earlier kernels
    grid_dep_launch();   // the fill's set-up overlaps; it waits for this grid's end
    if (rank == 0) {   // fresh counters for the fill and scan that follow
        if (tid == 0)
            w.ctr[CTR_ENTRIES] = w.ctr[CTR_OTICKET] = 0u;
        for (uint32_t i = tid; i < w.n_events; i += bd)
            w.ctr[CTR_EVENTS + i] = 0u;
    }
    for (uint32_t i = rank * bd + tid; i < w.n_seg; i += cs * bd)
        w.seg_peaks[i] = 0u;
    if (w.hit_off)
        for (uint32_t i = tid; i <= w.n_events; i += bd)
            s_off[i] = w.hit_off[i];
    __syncthreads();
    const uint32_t n = w.hit_off ? min(s_off[w.n_events], w.n_hits0) : w.n_hits0;
    uint32_t code[kBinClusterHPT], ev[kBinClusterHPT];
    float4 hv[kBinClusterHPT];   // x, y, z until the hit is binned
#pragma unroll
    for (uint32_t q = 0; q < kBinClusterHPT; ++q) {   // every hit's loads in flight
        const uint32_t h = (q * cs + rank) * bd + tid;
        hv[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (h < n)
            hv[q] = make_float4(__ldg(&w.x[h]), __ldg(&w.y[h]), __ldg(&w.z[h]), 0.0f);
    }
#pragma unroll
    for (uint32_t q = 0; q < kBinClusterHPT; ++q) {
        const uint32_t h = (q * cs + rank) * bd + tid;
        code[q] = kDropped;
        ev[q] = 0u;
        if (h < n) {
            const float x = hv[q].x, y = hv[q].y;
            float r2;
            code[q] = bin_code(g, et, ep, x, y, hv[q].z, r2);
            if (w.hit_off) {   // the last event whose first hit is <= h
                uint32_t lo = 0, hi = w.n_events - 1;
                while (lo < hi) {
                    const uint32_t mid = (lo + hi + 1) >> 1;
                    if (s_off[mid] <= h)
                        lo = mid;
                    else
                        hi = mid - 1;
                }
                ev[q] = lo;
            }
            hv[q] = make_float4(x, r2, __fmul_rn(2.0f, y), __uint_as_float(ev[q]));
            const uint32_t e = ev[q];
            for_each_slice(g, code[q], [&](uint32_t s) { atomicAdd(&s_cnt[e * g.n_slices + s], 1u); });
        }
    }
    // every CTA's counts are complete (and every CTA of the cluster runs); the
    // hits' lines are made while the others arrive
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    float2 line[kBinClusterHPT];
#pragma unroll
    for (uint32_t q = 0; q < kBinClusterHPT; ++q) {
        line[q] = make_float2(0.0f, 0.0f);
        if (code[q] != kDropped)
            line[q] = vote_line(g, hv[q].x, hv[q].y, hv[q].z);
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const uint32_t *r_cnt[kBinClusterMax];
#pragma unroll
    for (uint32_t r = 0; r < kBinClusterMax; ++r)
        r_cnt[r] = cl.map_shared_rank(s_cnt, r < cs ? r : 0u);
    for (uint32_t u = tid; u < U; u += bd) {
        uint32_t c[kBinClusterMax];
#pragma unroll
        for (uint32_t r = 0; r < kBinClusterMax; ++r)
            c[r] = r < cs ? r_cnt[r][u] : 0u;
        uint32_t tot = 0, below = 0;
#pragma unroll
        for (uint32_t r = 0; r < kBinClusterMax; ++r) {
            below += r < rank ? c[r] : 0u;
            tot += c[r];
        }
        s_tot[u] = tot;
        s_pl[u] = below;
    }
    // done with the other CTAs' counts: arrive now, wait before exiting, so
    // that every CTA's shared memory outlives every read of it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    __syncthreads();
    const uint32_t total = block_exclusive_scan(s_tot, U, s_wsum);   // totals -> unit offsets
    if (tid == 0)
        s_tot[U] = total;
    for (uint32_t u = tid; u < U; u += bd) {
        s_pl[u] += s_tot[u];   // this CTA's first list index in unit u
        if (rank == 0)
            w.slice_off[u] = s_tot[u];
    }
    if (rank == 0 && tid == 0)
        w.slice_off[U] = total;
    __syncthreads();
#pragma unroll
    for (uint32_t q = 0; q < kBinClusterHPT; ++q) {
        const uint32_t e = ev[q];
        for_each_slice(g, code[q], [&](uint32_t s) {
            const uint32_t idx = atomicAdd(&s_pl[e * g.n_slices + s], 1u);
            if (idx < w.list_cap) {
                w.list[idx] = hv[q];
                w.lines[idx] = line[q];
            }
        });
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// k_fill_priv
// ---------------------------------------------------------------------------
// Row swizzle inside 32-word blocks of the shared tile: spreads the banks
// of a warp whose lanes (consecutive A rows) vote into the same B column.
__device__ __forceinline__ uint32_t row_hash(uint32_t r)
{
    return (r * 0x9E3779B9u) >> 27;  // 5 bits
}

// Cells >= T of one pass: hot[] marks their rows (bit r of word r / 32),
// cand[] lists them as r * n_b + j (up to cap; *n counts them all), candv[]
// holds their votes where the lister knows them.
struct FlushList {
    uint32_t *hot;
    uint32_t *cand;     // r * n_b + j
    uint32_t *candv;    // the cell's votes
    uint32_t *n;
    uint32_t cap;
};

// Votes of hits hs[hl], hs[hl + hstride], .. < nc (the vote lines of the
// records rec[0 .. nc)) into tile row r (A bin i).
template <bool U16>
__device__ __forceinline__ void vote_rows(const Geom &g, uint32_t *tile, const float2 *hs, const float4 *rec,
                                          uint32_t nc, uint32_t r, uint32_t i, uint32_t hl, uint32_t hstride,
                                          uint32_t pitch)
{
    const uint32_t rowbase = r * pitch;
    const uint32_t sw = U16 ? (row_hash(r) & 0x1Eu) : (row_hash(r) & 0x1Cu);
#pragma unroll 4
    for (uint32_t h = hl; h < nc; h += hstride) {
        const uint32_t j = vote_bin_line(g, hs[h], i, rec + h);
        if (j < g.nb) {
            if (U16)
                atomicAdd(&tile[rowbase + ((j >> 1) ^ sw)], 1u << ((j & 1u) << 4));
            else
                atomicAdd(&tile[rowbase + (j ^ sw)], 1u);
        }
    }
}

template <bool LIST>
__device__ __forceinline__ void list_cells(const Geom &g, const FlushList &L, uint32_t r, uint32_t j0,
                                           const uint32_t *v, uint32_t n)
{
    if (!LIST)
        return;
    uint32_t mx = 0;
    for (uint32_t m = 0; m < n; ++m)
        mx = max(mx, v[m]);
    if (mx < g.threshold)
        return;
    atomicOr(&L.hot[r >> 5], 1u << (r & 31u));
    for (uint32_t m = 0; m < n; ++m)
        if (v[m] >= g.threshold) {
            const uint32_t p = atomicAdd(L.n, 1u);
            if (p < L.cap) {
                L.cand[p] = r * g.nb + j0 + m;
                L.candv[p] = v[m];
            }
        }
}

// Write tile rows r0 .. r0 + rows - 1 of one pass to dst (M_H, or with
// !GDST a shared-memory staging buffer, from its first row on) and clear
// them; with LIST, list the cells >= T (as pass rows r0 + r); with
// accumulate, add to M_H.
// The tile keeps row r's logical word w at physical word w ^ sw(r) (sw even
// in u16 mode, a multiple of 4 in u32 mode).  When n_b is a multiple of 4
// each step moves 4 cells: consecutive threads write consecutive 16-byte
// pieces of the row, so every store instruction of a warp covers 512
// contiguous bytes.
template <bool U16, bool LIST, bool ACC, class G = BlockGroup, bool GDST = true>
__device__ __forceinline__ void flush_tile(const Geom &g, uint32_t *tile, uint32_t *dst, uint32_t rows,
                                           uint32_t pitch, const FlushList &L, uint32_t r0 = 0)
{
    const uint32_t tid = G::rank(), bd = G::size(), nb = g.nb;
    // one 16-byte unit (4 cells) of row r0 + r, column group c4: read + clear
    // the tile words, write (or add to) the output at o, list the cells >= T
    auto unit = [&](uint32_t rl, uint32_t c4, uint4 *o) {
        const uint32_t r = r0 + rl;
        uint32_t v[4];
        if (U16) {
            uint2 *p = reinterpret_cast<uint2 *>(&tile[r * pitch + ((2u * c4) ^ (row_hash(r) & 0x1Eu))]);
            const uint2 pr = *p;
            *p = make_uint2(0u, 0u);
            v[0] = pr.x & 0xffffu; v[1] = pr.x >> 16; v[2] = pr.y & 0xffffu; v[3] = pr.y >> 16;
        } else {
            uint4 *p = reinterpret_cast<uint4 *>(&tile[r * pitch + ((4u * c4) ^ (row_hash(r) & 0x1Cu))]);
            const uint4 pr = *p;
            *p = make_uint4(0u, 0u, 0u, 0u);
            v[0] = pr.x; v[1] = pr.y; v[2] = pr.z; v[3] = pr.w;
        }
        if (ACC) {
            const uint4 old = *o;
            v[0] += old.x; v[1] += old.y; v[2] += old.z; v[3] += old.w;
        }
        // to M_H a streaming store (evict-first): M_H is written once per fill and
        // read back only at the candidates, so its lines should not displace
        // other data in L2; a staging buffer in shared memory takes a plain store
        if (GDST)
            __stcs(o, make_uint4(v[0], v[1], v[2], v[3]));
        else
            *o = make_uint4(v[0], v[1], v[2], v[3]);
        list_cells<LIST>(g, L, r, 4u * c4, v, 4);
    };
    if ((nb & 3u) == 0) {
        const uint32_t q = nb >> 2;  // 16-byte units per row
        if (bd % q == 0) {
            // the group covers whole rows: each thread keeps its column group
            // and steps down bd / q rows at a time
            const uint32_t rstep = bd / q, c4 = tid % q;
            uint4 *o = reinterpret_cast<uint4 *>(dst) + tid;
            for (uint32_t r = tid / q; r < rows; r += rstep, o += bd)
                unit(r, c4, o);
        } else {
            const uint32_t qs = (q & (q - 1)) ? 32u : (uint32_t)(__ffs(q) - 1);
            const uint32_t units = rows * q;
            for (uint32_t u = tid; u < units; u += bd) {
                const uint32_t r = qs < 32u ? u >> qs : u / q;
                unit(r, u - r * q, reinterpret_cast<uint4 *>(dst) + u);
            }
        }
    } else {
        const uint32_t units = rows * nb;
        for (uint32_t u = tid; u < units; u += bd) {
            const uint32_t rl = u / nb, j = u - rl * nb, r = r0 + rl;
            uint32_t v;
            if (U16) {
                const uint32_t word = r * pitch + ((j >> 1) ^ (row_hash(r) & 0x1Eu));
                v = (tile[word] >> ((j & 1u) << 4)) & 0xffffu;
            } else {
                const uint32_t word = r * pitch + (j ^ (row_hash(r) & 0x1Cu));
                v = tile[word];
            }
            v = ACC ? dst[u] + v : v;
            dst[u] = v;
            list_cells<LIST>(g, L, r, j, &v, 1);
        }
        G::sync();
        // clear the rows after every thread has read its cells
        for (uint32_t k = tid; k < rows * pitch; k += bd)
            tile[r0 * pitch + k] = 0u;
    }
}

// Copy up to cap vote lines of a unit's list, from list index pos on (pos
// < end), into hs; advances pos.  All threads of the group call it.
template <class G = BlockGroup>
__device__ __forceinline__ uint32_t stage_hits(const Work &w, float2 *hs, uint32_t cap, uint32_t &pos, uint32_t end)
{
    G::sync();   // the previous readers of hs are done
    const uint32_t n = min(cap, end - pos);
    constexpr uint32_t U = 4;
    for (uint32_t k0 = 0; k0 < n; k0 += U * G::size()) {
        float2 v[U];
#pragma unroll
        for (uint32_t q = 0; q < U; ++q) {
            const uint32_t k = k0 + q * G::size() + G::rank();
            if (k < n)
                v[q] = __ldg(&w.lines[pos + k]);
        }
#pragma unroll
        for (uint32_t q = 0; q < U; ++q) {
            const uint32_t k = k0 + q * G::size() + G::rank();
            if (k < n)
                hs[k] = v[q];
        }
    }
    pos += n;
    G::sync();
    return n;
}

// The votes of one strip pass: tile rows 0 .. pr - 1 are A bins i - r ..,
// from the hits of list entries l0 .. l1 of unit es.  Hits are staged HC at
// a time; when a unit's hits fit they stay staged for its later passes
// (cached_es / cached_n).  SYNC: a cached pass starts with a group barrier
// (the previous pass's readers of the tile are done); without it the caller
// orders the tile by other means.  All threads of the group call it.
template <class G, bool SYNC>
__device__ __forceinline__ void vote_pass(const Geom &g, const Work &w, uint32_t *tile, float2 *hs, uint32_t HC,
                                          uint64_t es, uint32_t l0, uint32_t l1, uint64_t &cached_es,
                                          uint32_t &cached_n, bool u16, uint32_t r, uint32_t pr, uint32_t i,
                                          uint32_t hl, uint32_t hstride, uint32_t pitch)
{
    if (cached_es == es) {
        if (SYNC)
            G::sync();
        if (r < pr) {
            if (u16)
                vote_rows<true>(g, tile, hs, w.list + l0, cached_n, r, i, hl, hstride, pitch);
            else
                vote_rows<false>(g, tile, hs, w.list + l0, cached_n, r, i, hl, hstride, pitch);
        }
        return;
    }
    cached_es = ~0ull;   // hs is about to be overwritten
    uint32_t pos = l0;
    bool first = true;
    while (first || pos < l1) {
        const float4 *rec = w.list + pos;
        const uint32_t nsel = stage_hits<G>(w, hs, HC, pos, l1);
        if (first && pos >= l1) {
            cached_es = es;   // the whole list fits: keep it
            cached_n = nsel;
        }
        first = false;
        if (r < pr) {
            if (u16)
                vote_rows<true>(g, tile, hs, rec, nsel, r, i, hl, hstride, pitch);
            else
                vote_rows<false>(g, tile, hs, rec, nsel, r, i, hl, hstride, pitch);
        }
    }
}

// The work items [it0, it1) of CTA `cta` of `grid`, counted from the first of
// the launch's units: the (event, slice, strip) items in order, cut where the estimated cost -- v = c.vote_weight
// per (hit, row) vote plus one per cell written -- reaches cta / grid of the
// total.  A unit u = (event, slice) costs n_a (n_b + v hits(u)), so the cost
// before unit u0 + u is n_a (n_b u + v (slice_off[u0 + u] - slice_off[u0])); a cut inside a unit falls
// on a strip boundary.  Every thread of the group calls
// it and gets the same result; s_res: 2 shared words.
template <class G = BlockGroup>
__device__ __forceinline__ void cta_items(const Geom &g, const Work &w, const FillCfg &c, uint32_t cta,
                                          uint32_t grid, uint64_t n_static, uint64_t &it0, uint64_t &it1,
                                          unsigned long long *s_res)
{
    const uint32_t U = w.nu, off0 = __ldcg(&w.slice_off[w.u0]);
    auto cost = [&](uint32_t u) {
        return (uint64_t)g.na *
               ((uint64_t)g.nb * u + (uint64_t)c.vote_weight * (__ldcg(&w.slice_off[w.u0 + u]) - off0));
    };
    // the cost of the first n_static items
    const uint32_t us = (uint32_t)(n_static / c.strips), ks = (uint32_t)(n_static % c.strips);
    uint64_t total = cost(us);
    if (ks)
        total += ks * ((cost(us + 1) - total + c.strips - 1) / c.strips);
    const uint64_t items = n_static;
    const uint64_t T0 = (total / grid) * cta + ((total % grid) * cta) / grid;
    const uint64_t T1 = (total / grid) * (cta + 1) + ((total % grid) * (cta + 1)) / grid;
    if (G::rank() == 0)
        s_res[0] = s_res[1] = items;
    G::sync();
    for (uint32_t u = G::rank(); u < U; u += G::size()) {
        const uint64_t a = cost(u), b = cost(u + 1);
        const uint64_t per = (b - a + c.strips - 1) / c.strips;   // one strip, rounded up
        const uint64_t last = c.strips - 1;
        if (a <= T0 && T0 < b) {
            const uint64_t k = (T0 - a) / per;
            s_res[0] = (uint64_t)u * c.strips + (k < last ? k : last);
        }
        if (a <= T1 && T1 < b) {
            const uint64_t k = (T1 - a) / per;
            s_res[1] = (uint64_t)u * c.strips + (k < last ? k : last);
        }
    }
    G::sync();
    it0 = min((uint64_t)s_res[0], items);
    it1 = cta + 1 == grid ? items : min((uint64_t)s_res[1], items);
    G::sync();   // s_res may be reused
}

// Hand out the next run-time item (see dyn_items): returns its rank, or
// n_dyn once none is left -- after which the last CTA to find none resets
// both counters for the next fill.  All threads of the block call it.
__device__ __forceinline__ uint32_t next_dyn_item(const Work &w, uint32_t n_dyn, uint32_t *s_word)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t d = n_dyn;
        if (n_dyn)
            d = atomicAdd(&w.ctr[CTR_DYN], 1u);
        if (d >= n_dyn) {
            d = n_dyn;
            __threadfence();
            if (atomicAdd(&w.ctr[CTR_DYN_DONE], 1u) == gridDim.x - 1) {
                w.ctr[CTR_DYN] = 0u;
                w.ctr[CTR_DYN_DONE] = 0u;
            }
        }
        *s_word = d;
    }
    __syncthreads();
    return *s_word;
}

// Walks the (event, slice, strip) work items it0, it0 + 1, ... of a CTA with
// one 64-bit decomposition at the start and carries afterwards (a 64-bit
// division per item and thread costs more than a strip's flush setup).
struct ItemCursor {
    uint32_t k, s, e;   // strip, slice, event
    uint64_t es;        // e * n_slices + s
    __device__ __forceinline__ ItemCursor(const Geom &g, const FillCfg &c, uint64_t item)
    {
        k = (uint32_t)(item % c.strips);
        es = item / c.strips;
        s = (uint32_t)(es % g.n_slices);
        e = (uint32_t)(es / g.n_slices);
    }
    __device__ __forceinline__ void next(const Geom &g, const FillCfg &c)
    {
        if (++k == c.strips) {
            k = 0;
            ++es;
            if (++s == g.n_slices) {
                s = 0;
                ++e;
            }
        }
    }
};

__global__ void __launch_bounds__(1024) k_fill_priv(Geom g, Work w, FillCfg c)
{
    extern __shared__ uint4 sm4[];
    uint32_t *tile = reinterpret_cast<uint32_t *>(sm4);
    float2 *hs = reinterpret_cast<float2 *>(tile + c.tile_words);

    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    for (uint32_t k = tid; k < c.tile_words / 4; k += bd)
        sm4[k] = make_uint4(0u, 0u, 0u, 0u);
    grid_dep_wait();   // the unit lists of k_scatter

    __shared__ unsigned long long s_rng[2];
    __shared__ uint32_t s_dyn;
    const uint64_t items = (uint64_t)w.nu * c.strips, first = (uint64_t)w.u0 * c.strips;
    const uint64_t n_dyn = c.dyn ? dyn_items(items, gridDim.x) : 0, n_static = items - n_dyn;
    uint64_t it0, it1;
    cta_items(g, w, c, blockIdx.x, gridDim.x, n_static, it0, it1, s_rng);
    uint64_t cached_es = ~0ull;   // (event, slice) whose whole hit list is in hs
    uint32_t cached_n = 0;

    auto do_item = [&](const ItemCursor &cur) {
        const uint32_t k = cur.k;
        const uint64_t es = cur.es;
        const uint32_t s = cur.s;
        const uint32_t e = cur.e;
        const uint32_t l0 = __ldg(&w.slice_off[es]), l1 = __ldg(&w.slice_off[es + 1]);   // the unit's hits
        const uint32_t i0 = k * c.W;
        const uint32_t rows = min(c.W, g.na - i0);
        // u16 counters are exact while the slice holds < 65536 hits
        const bool u16 = (l1 - l0) < 65536u;
        const uint32_t rpass = u16 ? c.W : c.W / 2;
        const uint32_t pitch = u16 ? c.pitch16 : c.pitch32;
        uint32_t *Mrow = w.M + (size_t)e * w.n_cells + ((size_t)s * g.na + i0) * g.nb;
        const uint32_t r = tid % rpass, hl = tid / rpass, hstride = bd / rpass;

        for (uint32_t p0 = 0; p0 < rows; p0 += rpass) {
            const uint32_t pr = min(rpass, rows - p0);
            const uint32_t i = i0 + p0 + r;
            vote_pass<BlockGroup, true>(g, w, tile, hs, c.HC, es, l0, l1, cached_es, cached_n, u16, r, pr,
                                               i, hl, hstride, pitch);
            __syncthreads();
            uint32_t *dst = Mrow + (size_t)p0 * g.nb;
            if (c.accumulate) {
                if (u16)
                    flush_tile<true, false, true>(g, tile, dst, pr, pitch, FlushList{});
                else
                    flush_tile<false, false, true>(g, tile, dst, pr, pitch, FlushList{});
            } else {
                if (u16)
                    flush_tile<true, false, false>(g, tile, dst, pr, pitch, FlushList{});
                else
                    flush_tile<false, false, false>(g, tile, dst, pr, pitch, FlushList{});
            }
        }
    };
    ItemCursor cur(g, c, first + it0);
    for (uint64_t item = it0; item < it1; ++item, cur.next(g, c))
        do_item(cur);
    if (c.dyn)
        for (uint32_t d; (d = next_dyn_item(w, (uint32_t)n_dyn, &s_dyn)) < n_dyn;)
            do_item(ItemCursor(g, c, first + n_static + d));
}

// ---------------------------------------------------------------------------
// k_copy: M_H into a caller's device memory, a CTA per piece of it, 32 bytes
// per load.  Bound by the writes: M_H is compressed where it is sparse, so most
// reads never reach HBM.  The paper's matrix (268 MB, 4 % of the cells with
// votes): 55.5 us, in plain memory 82.2 us (cudaMemcpyAsync: 69.3 and 86.3 us;
// 16-byte loads 57.6 us, four CTAs per SM that go over the whole 63.7 us).
// ---------------------------------------------------------------------------
constexpr uint32_t kCopyThreads = 512;

struct Cells8 {
    uint32_t v[8];
};

__device__ __forceinline__ Cells8 load8(const uint32_t *p)
{
    Cells8 c;
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(c.v[0]), "=r"(c.v[1]), "=r"(c.v[2]), "=r"(c.v[3]), "=r"(c.v[4]), "=r"(c.v[5]), "=r"(c.v[6]),
                   "=r"(c.v[7])
                 : "l"(p)
                 : "memory");
    return c;
}

__device__ __forceinline__ void store8(uint32_t *p, const Cells8 &c)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(c.v[0]), "r"(c.v[1]),
                 "r"(c.v[2]), "r"(c.v[3]), "r"(c.v[4]), "r"(c.v[5]), "r"(c.v[6]), "r"(c.v[7])
                 : "memory");
}

// src and dst: 32-byte aligned
__global__ void __launch_bounds__(kCopyThreads) k_copy(uint32_t *dst, const uint32_t *src, uint64_t n)
{
    grid_dep_wait();
    const uint64_t n8 = n / 8u, i = (uint64_t)blockIdx.x * (2u * kCopyThreads) + threadIdx.x, k = i + kCopyThreads;
    Cells8 a, b;
    if (i < n8)
        a = load8(src + 8u * i);
    if (k < n8)
        b = load8(src + 8u * k);
    if (i < n8)
        store8(dst + 8u * i, a);
    if (k < n8)
        store8(dst + 8u * k, b);
    if (blockIdx.x == 0 && threadIdx.x < (n & 7u))
        dst[8u * n8 + threadIdx.x] = src[8u * n8 + threadIdx.x];
}

// ---------------------------------------------------------------------------
// Naive path (the paper's CUDA fill): clear + global atomics.
// ---------------------------------------------------------------------------
__global__ void k_clear(uint32_t *M, uint64_t words)
{
    grid_dep_wait();
    const uint64_t n4 = words >> 2;
    uint4 *M4 = reinterpret_cast<uint4 *>(M);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n4; k += stride)
        M4[k] = make_uint4(0u, 0u, 0u, 0u);
    for (uint64_t k = (n4 << 2) + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < words; k += stride)
        M[k] = 0u;
}

// The unit (event, slice) of hit record rec of the (event, slice) lists: the
// largest u' <= u with slice_off[u'] <= rec (slice_off[0] = 0), found by the
// warp 32 units at a time.  Every lane returns it; the whole warp calls it.
__device__ __forceinline__ uint32_t unit_below(const uint32_t *slice_off, uint32_t u, uint32_t rec)
{
    const uint32_t lane = threadIdx.x & 31u;
    for (;;) {
        const bool ok = lane <= u && __ldg(&slice_off[u - lane]) <= rec;
        const uint32_t m = __ballot_sync(0xffffffffu, ok);
        if (m)
            return u - (uint32_t)(__ffs(m) - 1);
        if (u < 32u)
            return 0u;
        u -= 32u;
    }
}

// The paper's fill (Sec. 3): a 1-D grid over hits, a thread block over A,
// one global atomicAdd per vote.  The hits come from k_scatter's (event,
// slice) lists, one (hit, slice) record per block at a time, and the grid
// (what the GPU holds at once) strides over the records from the last to
// the first: the blocks in flight work on neighbouring records, so their
// votes land in a few slices of M_H that stay in L2, and the first slices
// voted are the last ones the clear wrote.  The B bin comes from the
// threshold table in shared memory when it fits (48 KB), else from the
// division rule; both give the same bin for every B.
__global__ void __launch_bounds__(1024, 2) k_fill_naive(Geom g, Work w)
{
    extern __shared__ float s_beta[];   // n_b + 1 B-bin thresholds, or none
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    const bool tab = ((size_t)g.nb + 1) * 4 <= 48u * 1024u;
    if (tab)
        for (uint32_t k = tid; k <= g.nb; k += bd)
            s_beta[k] = g.bth[k];
    __syncthreads();
    grid_dep_wait();
    const float b_lo = tab ? s_beta[0] : 0.0f, b_hi = tab ? s_beta[g.nb] : 0.0f;
    const uint32_t U = w.n_events * g.n_slices;
    if (U == 0)
        return;
    const uint32_t n_rec = min(__ldg(&w.slice_off[U]), w.list_cap);
    const uint64_t slice_cells = (uint64_t)g.na * g.nb;
    uint32_t u = U - 1u;
    for (uint32_t k = blockIdx.x; k < n_rec; k += gridDim.x) {
        const uint32_t rec = n_rec - 1u - k;
        u = unit_below(w.slice_off, u, rec);
        const float4 hv = w.list[rec];
        const uint32_t e = u / g.n_slices, s = u - e * g.n_slices;
        uint32_t *Ms = w.M + (size_t)e * w.n_cells + (size_t)s * slice_cells;
        for (uint32_t i = tid; i < g.na; i += bd) {
            const float twoA = __fmul_rn(2.0f, a_centre(g, i));
            const int j = tab ? vote_bin_tab(g, s_beta, b_lo, b_hi, twoA, hv.x, hv.y, hv.z)
                              : vote_bin(g, twoA, hv.x, hv.y, hv.z);
            if (j >= 0)
                atomicAdd(&Ms[(size_t)i * g.nb + (uint32_t)j], 1u);
        }
    }
}

// ---------------------------------------------------------------------------
// Scan
// ---------------------------------------------------------------------------
// Peak test of the cell at column j of `row` (value v >= threshold).
// up / dn are the neighbouring rows of the same slice or nullptr.
__device__ __forceinline__ bool is_peak(const uint32_t *row, const uint32_t *up, const uint32_t *dn,
                                        uint32_t j, uint32_t nb, uint32_t v)
{
    const bool hl = j > 0, hr = j + 1 < nb;
    if (up) {
        if (hl && !(v > up[j - 1])) return false;
        if (!(v > up[j])) return false;
        if (hr && !(v > up[j + 1])) return false;
    }
    if (hl && !(v > row[j - 1])) return false;
    if (hr && !(v >= row[j + 1])) return false;
    if (dn) {
        if (hl && !(v >= dn[j - 1])) return false;
        if (!(v >= dn[j])) return false;
        if (hr && !(v >= dn[j + 1])) return false;
    }
    return true;
}

struct ScanSmem {
    uint32_t wsum[40];
    uint32_t round_total;
    uint32_t chunk_base;
    uint32_t abort;
    uint32_t pad;
};

// Where a CTA (or a handed-out fill item) registers its chunks: its row of
// a.desc, seq_max entries.
struct ChunkList {
    uint2 *desc;
    uint32_t cap;
};

__device__ __forceinline__ ChunkList interior_list(const ScanArgs &a, uint32_t cta)
{
    return ChunkList{a.desc + (size_t)cta * a.seq_max, a.seq_max};
}

// Flush the CTA's buffered peaks as one chunk of list L.
template <class G = BlockGroup>
__device__ __forceinline__ void flush_chunk(const ScanArgs &a, ScanSmem &ss, const uint4 *pbuf,
                                            uint32_t &buf_n, uint32_t &nseq, const ChunkList &L,
                                            uint32_t *status)
{
    if (buf_n == 0)
        return;
    if (G::rank() == 0) {
        ss.chunk_base = atomicAdd(a.g_count, buf_n);
        if (nseq < L.cap)
            L.desc[nseq] = make_uint2(ss.chunk_base, buf_n);
        if (nseq >= L.cap || ss.chunk_base + buf_n > a.entries_cap)
            atomicOr(status, (uint32_t)ST_SCRATCH_OVERFLOW);
    }
    G::sync();
    const uint32_t base = ss.chunk_base;
    for (uint32_t k = G::rank(); k < buf_n; k += G::size())
        if (base + k < a.entries_cap)
            a.entries[base + k] = pbuf[k];
    nseq += 1;
    buf_n = 0;
    G::sync();
}

// Ordered compaction of one round: each thread holds cnt peaks in pj/pv
// (columns of the row starting at row_lin0); appends them to pbuf in
// thread order and counts them for their event.
template <class G = BlockGroup, bool COUNT = true>
__device__ __forceinline__ void compact_round(ScanSmem &ss, uint4 *pbuf, uint32_t &buf_n, uint32_t cnt,
                                              const uint32_t *pj, const uint32_t *pv, uint32_t row_lin0,
                                              uint32_t event, uint32_t *ev_count)
{
    const uint32_t tid = G::rank(), warp = tid >> 5, lane = tid & 31u;
    const uint32_t nw = (G::size() + 31) >> 5;
    const uint32_t incl = warp_incl_scan(cnt);
    if (lane == 31u)
        ss.wsum[warp] = incl;
    G::sync();
    if (warp == 0) {
        const uint32_t v = lane < nw ? ss.wsum[lane] : 0u;
        const uint32_t vi = warp_incl_scan(v);
        ss.wsum[lane] = vi - v;
        if (lane == 31u) {
            ss.round_total = vi;
            if (COUNT)
                atomicAdd(&ev_count[event], vi);
        }
    }
    G::sync();
    const uint32_t pos = buf_n + ss.wsum[warp] + incl - cnt;
    for (uint32_t k = 0; k < cnt; ++k)
        pbuf[pos + k] = make_uint4(row_lin0 + pj[k], event, pv[k], 0u);
    buf_n += ss.round_total;
    G::sync();
}

// Ordered compaction of one entry per thread (has = 0 or 1): appends the
// entries to pbuf in thread order and counts them for their events.
template <class G = BlockGroup, bool COUNT = true>
__device__ __forceinline__ void compact_entry(ScanSmem &ss, uint4 *pbuf, uint32_t &buf_n, uint32_t has,
                                              const uint4 &ent, uint32_t *ev_count)
{
    const uint32_t tid = G::rank(), warp = tid >> 5, lane = tid & 31u;
    const uint32_t nw = (G::size() + 31) >> 5;
    const uint32_t incl = warp_incl_scan(has);
    if (lane == 31u)
        ss.wsum[warp] = incl;
    G::sync();
    if (warp == 0) {
        const uint32_t v = lane < nw ? ss.wsum[lane] : 0u;
        const uint32_t vi = warp_incl_scan(v);
        ss.wsum[lane] = vi - v;
        if (lane == 31u)
            ss.round_total = vi;
    }
    G::sync();
    if (has) {
        pbuf[buf_n + ss.wsum[warp] + incl - 1] = ent;
        if (COUNT)
            atomicAdd(&ev_count[ent.y], 1u);
    }
    buf_n += ss.round_total;
    G::sync();
}

// Detailed pass over global rows [ra, rb): candidates, neighbour tests and
// ordered compaction.  Rows [ra - 1, rb + 1) (clipped) are readable at
// base + (gr - b_first) * nb.  Each thread takes VEC consecutive cells.
template <int VEC>
__device__ void scan_rows_slow(const Geom &g, const Work &w, const ScanArgs &a, ScanSmem &ss, uint4 *pbuf,
                               uint32_t &buf_n, uint32_t &nseq, uint32_t &total, uint64_t ra, uint64_t rb,
                               const uint32_t *base, uint64_t b_first)
{
    const uint32_t tid = threadIdx.x, bd = blockDim.x, nb = g.nb, T = g.threshold;
    const uint64_t rows_ev = (uint64_t)g.n_slices * g.na;
    const uint32_t units = nb / VEC;
    const uint32_t rounds = (units + bd - 1) / bd;
    for (uint64_t gr = ra; gr < rb; ++gr) {
        const uint32_t i = (uint32_t)(gr % g.na);
        const uint64_t row_all = gr + (uint64_t)w.u0 * g.na;   // of all matrices' rows
        const uint32_t ev = (uint32_t)(row_all / rows_ev);
        const uint32_t row_lin0 = (uint32_t)((row_all - (uint64_t)ev * rows_ev) * nb);
        const uint32_t *row = base + (gr - b_first) * nb;
        const uint32_t *up = i > 0 ? row - nb : nullptr;
        const uint32_t *dn = i + 1 < g.na ? row + nb : nullptr;
        for (uint32_t rd = 0; rd < rounds; ++rd) {
            const uint32_t u = rd * bd + tid;
            uint32_t cnt = 0, pj[VEC], pv[VEC];
            if (u < units) {
#pragma unroll
                for (uint32_t c = 0; c < (uint32_t)VEC; ++c) {
                    const uint32_t j = VEC * u + c;
                    const uint32_t v = row[j];
                    if (v >= T && is_peak(row, up, dn, j, nb, v)) {
                        pj[cnt] = j;
                        pv[cnt] = v;
                        ++cnt;
                    }
                }
            }
            if (__syncthreads_or(cnt)) {
                // at most 2 peaks among 4 consecutive cells (no two peaks are neighbours)
                if (buf_n + (VEC > 1 ? 2u : 1u) * bd > a.K)
                    flush_chunk(a, ss, pbuf, buf_n, nseq, interior_list(a, blockIdx.x), w.status);
                compact_round(ss, pbuf, buf_n, cnt, pj, pv, row_lin0, ev, a.ev_count);
                total += ss.round_total;
            }
        }
    }
}

// TMA-staged scan (n_b % 4 == 0).
__global__ void __launch_bounds__(256) k_scan_tma(Geom g, Work w, ScanArgs a)
{
    grid_dep_wait();
    extern __shared__ uint4 sm4[];
    // layout: [0, 192) ScanSmem | [192, 256) 8 mbarriers | K peak entries | S stage slots
    ScanSmem &ss = *reinterpret_cast<ScanSmem *>(sm4);
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm4 + 12);
    uint4 *pbuf = sm4 + 16;
    uint32_t *slots = reinterpret_cast<uint32_t *>(pbuf + a.K);

    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    const uint32_t nb = g.nb, T = g.threshold;
    const uint64_t G = (uint64_t)g.na * w.nu;
    const uint64_t g0 = G * blockIdx.x / gridDim.x, g1 = G * (blockIdx.x + 1) / gridDim.x;
    const uint32_t R = a.R, S = a.S;
    const uint64_t n_stages = (g1 - g0 + R - 1) / R;
    uint32_t buf_n = 0, nseq = 0, total = 0;

    if (tid == 0) {
        ss.abort = 0;
        for (uint32_t q = 0; q < S; ++q)
            mbar_init(&bars[q], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // stage k: own rows [g0 + kR, min(g0 + (k+1)R, g1)), loaded with one
    // halo row on each side (clipped to the matrix).
    auto issue = [&](uint64_t k) {
        const uint64_t ra = g0 + k * R, rb = min(ra + R, g1);
        const uint64_t ba = ra > 0 ? ra - 1 : 0, bb = min(rb + 1, G);
        const uint32_t q = (uint32_t)(k % S);
        const uint32_t bytes = (uint32_t)((bb - ba) * nb * 4u);
        mbar_arrive_expect_tx(&bars[q], bytes);
        bulk_load(slots + (size_t)q * a.slot_words, w.M + ba * nb, bytes, &bars[q]);
    };
    if (tid == 0)
        for (uint64_t k = 0; k < n_stages && k < S; ++k)
            issue(k);

    uint64_t k_abort = 0;
    for (uint64_t k = 0; k < n_stages; ++k) {
        const uint64_t ra = g0 + k * R, rb = min(ra + R, g1);
        const uint64_t ba = ra > 0 ? ra - 1 : 0;
        const uint32_t q = (uint32_t)(k % S);
        const uint32_t *slot = slots + (size_t)q * a.slot_words;
        if (!mbar_wait_bounded(&bars[q], (uint32_t)((k / S) & 1u)))
            atomicOr(&ss.abort, 1u);
        __syncthreads();
        if (ss.abort) {
            k_abort = k;
            break;
        }
        // fast path: any cell >= T among the stage's own rows?
        const uint4 *own = reinterpret_cast<const uint4 *>(slot + (ra - ba) * nb);
        const uint32_t n4 = (uint32_t)(rb - ra) * (nb >> 2);
        uint32_t hot = 0;
        for (uint32_t u = tid; u < n4; u += bd) {
            const uint4 v = own[u];
            hot |= (max(max(v.x, v.y), max(v.z, v.w)) >= T);
        }
        if (__syncthreads_or(hot))
            scan_rows_slow<4>(g, w, a, ss, pbuf, buf_n, nseq, total, ra, rb, slot, ba);
        __syncthreads();  // every thread is done with slot q
        if (tid == 0 && k + S < n_stages) {
            fence_proxy_async_smem();
            issue(k + S);
        }
    }
    if (ss.abort) {
        // let the copies still in flight (bounded wait) land before the CTA exits
        if (tid == 0) {
            atomicOr(w.status, (uint32_t)ST_WAIT_TIMEOUT);
            const uint64_t k_end = min(n_stages, k_abort + S);
            for (uint64_t kk = k_abort; kk < k_end; ++kk)
                (void)mbar_wait_bounded(&bars[kk % S], (uint32_t)((kk / S) & 1u));
        }
        __syncthreads();
    }
    flush_chunk(a, ss, pbuf, buf_n, nseq, interior_list(a, blockIdx.x), w.status);
    if (tid == 0) {
        a.cta_nseq[blockIdx.x] = min(nseq, a.seq_max);
        a.cta_total[blockIdx.x] = total;
    }
}

// Direct-load scan for any n_b (no staging).
__global__ void __launch_bounds__(256) k_scan_direct(Geom g, Work w, ScanArgs a)
{
    grid_dep_wait();
    extern __shared__ uint4 sm4[];
    ScanSmem &ss = *reinterpret_cast<ScanSmem *>(sm4);
    uint4 *pbuf = sm4 + 16;
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    const uint32_t nb = g.nb, T = g.threshold;
    const uint64_t G = (uint64_t)g.na * w.nu;
    const uint64_t g0 = G * blockIdx.x / gridDim.x, g1 = G * (blockIdx.x + 1) / gridDim.x;
    const uint32_t R = a.R;
    uint32_t buf_n = 0, nseq = 0, total = 0;
    for (uint64_t ra = g0; ra < g1; ra += R) {
        const uint64_t rb = min(ra + R, g1);
        const uint32_t *own = w.M + ra * nb;
        const uint64_t n = (rb - ra) * nb;
        uint32_t hot = 0;
        for (uint64_t u = tid; u < n; u += bd)
            hot |= own[u] >= T;
        if (__syncthreads_or(hot))
            scan_rows_slow<1>(g, w, a, ss, pbuf, buf_n, nseq, total, ra, rb, w.M, 0);
    }
    flush_chunk(a, ss, pbuf, buf_n, nseq, interior_list(a, blockIdx.x), w.status);
    if (tid == 0) {
        a.cta_nseq[blockIdx.x] = min(nseq, a.seq_max);
        a.cta_total[blockIdx.x] = total;
    }
}

// ---------------------------------------------------------------------------
// The fused fill: Step 1 plus the first half of Step 2.
//
// Like k_fill_priv, a CTA owns a contiguous range of (event, slice, strip)
// items, votes each strip pass into a shared-memory tile and writes it to
// M_H, clearing the tile as it goes.  While writing, it lists the cells of
// the pass that hold >= T votes and appends them, in linear order, to its
// chunks of candidate entries -- the cells a full scan would have to look
// at.  k_peaks then tests only those candidates against their neighbours,
// once the whole of M_H is written (no row waits for another CTA), and
// compacts each chunk in place to the peaks; k_order places the chunks.
// A pass listing more than kFusedCand cells emits its rows' cells >= T from
// M_H instead (read back through L2).
// ---------------------------------------------------------------------------

// Peak test with the neighbours read through L2; up / dn are null outside
// the slice.  All eight loads are issued before any comparison, so a test
// costs one memory latency.
__device__ __forceinline__ bool is_peak_l2(const uint32_t *row, const uint32_t *up, const uint32_t *dn, uint32_t j,
                                           uint32_t nb, uint32_t v)
{
    const bool hl = j > 0, hr = j + 1 < nb;
    const uint32_t ul = up && hl ? __ldcg(up + j - 1) : 0u, uc = up ? __ldcg(up + j) : 0u,
                   ur = up && hr ? __ldcg(up + j + 1) : 0u;
    const uint32_t rl = hl ? __ldcg(row + j - 1) : 0u, rr = hr ? __ldcg(row + j + 1) : 0u;
    const uint32_t dl = dn && hl ? __ldcg(dn + j - 1) : 0u, dc = dn ? __ldcg(dn + j) : 0u,
                   dr = dn && hr ? __ldcg(dn + j + 1) : 0u;
    // absent neighbours read as 0: v > 0 and v >= 0 hold for every v >= 1
    return v > ul && v > uc && v > ur && v > rl && v >= rr && v >= dl && v >= dc && v >= dr;
}

// Append the candidate cells of one pass (rows iA .. iA + pr - 1 of slice
// unit `slice_lin0`) to the CTA's candidate chunks, in linear order.  n_c
// cells were listed as r * n_b + j in cand / candv (up to kFusedCand); with
// more, the rows marked in hotm are read back: pass row r from rowsA + r n_b
// when r < split, else from rowsB + (r - split) n_b -- M_H in global memory,
// or (SMEM) the shared staging buffers.  Entries are {lin within event,
// event, votes, 0}.  All threads of the group call it.
template <class G, bool SMEM = false>
__device__ __forceinline__ void emit_pass(const Geom &g, const Work &w, const ScanArgs &a, ScanSmem &ss, uint4 *pbuf,
                                          uint32_t &buf_n, uint32_t &nseq, uint32_t &total, const ChunkList &inner,
                                          const uint32_t *cand, const uint32_t *candv, uint32_t *srt, uint32_t *srtv,
                                          uint32_t n_c, uint64_t hotm, uint32_t pr, uint32_t iA, uint32_t slice_lin0,
                                          uint32_t e, const uint32_t *rowsA, const uint32_t *rowsB, uint32_t split)
{
    const uint32_t tid = G::rank(), bd = G::size(), nb = g.nb;
    const uint32_t lin0 = slice_lin0 + iA * nb;
    if (n_c <= 32u) {
        // few candidates: the first warp ranks them and writes them in order
        if (buf_n + n_c > a.K)
            flush_chunk<G>(a, ss, pbuf, buf_n, nseq, inner, w.status);
        if (tid < n_c) {
            const uint32_t key = cand[tid];
            uint32_t rank = 0;
            for (uint32_t m = 0; m < n_c; ++m)
                rank += cand[m] < key;
            pbuf[buf_n + rank] = make_uint4(lin0 + key, e, candv[tid], 0u);
        }
        buf_n += n_c;
        total += n_c;
        return;   // the caller's barrier follows before pbuf or the lists are used again
    }
    if (n_c <= kFusedCand) {
        // distinct keys: the rank of a key is the number of smaller ones
        for (uint32_t k = tid; k < n_c; k += bd) {
            const uint32_t key = cand[k];
            uint32_t rank = 0;
            for (uint32_t m = 0; m < n_c; ++m)
                rank += cand[m] < key;
            srt[rank] = key;
            srtv[rank] = candv[k];
        }
        // the sorted list is dense: append it to the chunk buffer as it is
        // (n_c <= kFusedCand <= K; a chunk is flushed with more than
        // K - kFusedCand entries, so the chunk bound of the rounds below holds)
        if (buf_n + n_c > a.K)
            flush_chunk<G>(a, ss, pbuf, buf_n, nseq, inner, w.status);   // its barriers order srt / srtv too
        else
            G::sync();
        for (uint32_t k = tid; k < n_c; k += bd)
            pbuf[buf_n + k] = make_uint4(lin0 + srt[k], e, srtv[k], 0u);
        buf_n += n_c;
        total += n_c;
        return;   // the caller's barrier follows before pbuf or the lists are used again
    }
    // rounds of rc threads, like the candidate rounds: a chunk is flushed
    // only when fewer than rc entries are free
    const uint32_t T = g.threshold, per_round = fused_round(bd, a.K);
    for (uint32_t r = 0; r < pr; ++r) {
        if (!((hotm >> r) & 1ull))
            continue;
        const uint32_t *row = r < split ? rowsA + (size_t)r * nb : rowsB + (size_t)(r - split) * nb;
        for (uint32_t j0 = 0; j0 < nb; j0 += per_round) {
            const uint32_t j = j0 + tid;
            uint32_t cnt = 0, pj[1], pv[1];
            if (tid < per_round && j < nb) {
                const uint32_t v = SMEM ? row[j] : __ldcg(row + j);
                if (v >= T) {
                    pj[0] = j;
                    pv[0] = v;
                    cnt = 1;
                }
            }
            if (G::sync_or(cnt)) {
                if (buf_n + per_round > a.K)
                    flush_chunk<G>(a, ss, pbuf, buf_n, nseq, inner, w.status);
                compact_round<G, false>(ss, pbuf, buf_n, cnt, pj, pv, lin0 + r * nb, e, nullptr);
                total += ss.round_total;
            }
        }
    }
}

// Write one pass from the tile to M_H, clear the tile, and emit its
// candidates (emit_pass).  empty_bar: arrived on once the tile is clear
// (the warp-specialised fill), or null.  All threads of the group call it.
template <class G, bool U16>
__device__ __forceinline__ void flush_emit_pass(const Geom &g, const Work &w, const ScanArgs &a, ScanSmem &ss,
                                                uint4 *pbuf, uint32_t &buf_n, uint32_t &nseq, uint32_t &total,
                                                const ChunkList &inner, uint32_t *tile, uint32_t pitch, uint32_t *dst,
                                                uint32_t pr, uint32_t iA, uint32_t slice_lin0, uint32_t e,
                                                const uint32_t *Ms, uint32_t *lists, uint32_t *s_hot, uint32_t *s_nc,
                                                uint64_t *empty_bar)
{
    uint32_t *cand = lists, *candv = lists + kFusedCand, *srt = lists + 2 * kFusedCand, *srtv = lists + 3 * kFusedCand;
    if (G::rank() == 0)
        s_hot[0] = s_hot[1] = *s_nc = 0u;
    G::sync();   // the pass's votes are complete (and the counters zero)
    flush_tile<U16, true, false, G>(g, tile, dst, pr, pitch, FlushList{s_hot, cand, candv, s_nc, kFusedCand});
    if (empty_bar)
        mbar_arrive(empty_bar);   // the tile is clear
    G::sync();                    // M_H rows of the pass and the lists visible to the group
    const uint64_t hotm = (uint64_t)s_hot[0] | ((uint64_t)s_hot[1] << 32);
    const uint32_t n_c = *s_nc;
    if (n_c)
        emit_pass<G>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, cand, candv, srt, srtv, n_c, hotm, pr, iA,
                     slice_lin0, e, Ms + (size_t)iA * g.nb, nullptr, pr);
    G::sync();                    // lists and counters free for the next pass
}

// The same through the u32 staging buffers stg[0], stg[1] (hrows rows of
// n_b cells each; k_fill_bulk): the pass leaves in halves of hrows rows.
// Each half waits until the bulk copy that last read its buffer is done
// (thread 0's async-groups, all but the newest), is converted into the
// buffer while the candidates are listed, and is copied to M_H by thread 0
// with one bulk copy (the half's rows are contiguous in the buffer and in
// M_H); the threads then go on while the copy drains.  *bsel alternates the
// buffers across halves.  Hot rows of an overflowing pass are read back
// from the buffers.  dst: the pass's first M_H row.  All threads of the
// block call it.
template <bool U16>
__device__ __forceinline__ void bulk_flush_emit_pass(const Geom &g, const Work &w, const ScanArgs &a, ScanSmem &ss,
                                                     uint4 *pbuf, uint32_t &buf_n, uint32_t &nseq, uint32_t &total,
                                                     const ChunkList &inner, uint32_t *tile, uint32_t pitch,
                                                     uint32_t *dst, uint32_t pr, uint32_t iA, uint32_t slice_lin0,
                                                     uint32_t e, uint32_t *stg, uint32_t hrows, uint32_t &bsel,
                                                     uint32_t *lists, uint32_t *s_hot, uint32_t *s_nc)
{
    uint32_t *cand = lists, *candv = lists + kFusedCand, *srt = lists + 2 * kFusedCand, *srtv = lists + 3 * kFusedCand;
    const uint32_t tid = threadIdx.x, nb = g.nb;
    if (tid == 0)
        s_hot[0] = s_hot[1] = *s_nc = 0u;
    const uint32_t b0 = bsel;   // the first half's buffer; the second takes the other
    for (uint32_t h0 = 0; h0 < pr; h0 += hrows) {
        const uint32_t nr = min(hrows, pr - h0);
        uint32_t *S = stg + (size_t)bsel * hrows * nb;
        if (tid == 0)
            bulk_wait_read<1>();   // the copy that last read buffer bsel is done
        __syncthreads();           // (first half: the votes and the counter reset are done too)
        flush_tile<U16, true, false, BlockGroup, false>(g, tile, S, nr, pitch,
                                                        FlushList{s_hot, cand, candv, s_nc, kFusedCand}, h0);
        fence_proxy_async_smem();  // the buffer's generic writes, visible to the bulk copies
        __syncthreads();
        if (tid == 0) {
            bulk_store(dst + (size_t)h0 * nb, S, nr * nb * 4u);
            bulk_commit();
        }
        bsel ^= 1u;
    }
    const uint64_t hotm = (uint64_t)s_hot[0] | ((uint64_t)s_hot[1] << 32);
    const uint32_t n_c = *s_nc;
    if (n_c)
        emit_pass<BlockGroup, true>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, cand, candv, srt, srtv, n_c, hotm,
                                    pr, iA, slice_lin0, e, stg + (size_t)b0 * hrows * nb,
                                    stg + (size_t)(b0 ^ 1u) * hrows * nb, hrows);
    __syncthreads();               // lists and counters free for the next pass
}

// The CTA's candidate bookkeeping once its range is done.
template <class G>
__device__ __forceinline__ void finish_candidates(const Work &w, const ScanArgs &a, ScanSmem &ss, const uint4 *pbuf,
                                                  uint32_t &buf_n, uint32_t &nseq, uint32_t total,
                                                  const ChunkList &inner, uint32_t cta)
{
    flush_chunk<G>(a, ss, pbuf, buf_n, nseq, inner, w.status);
    if (G::rank() == 0) {
        a.cta_nseq[cta] = min(nseq, a.seq_max);
        a.cta_total[cta] = total;
    }
}

// The body of both fused fills.  BULK (k_fill_bulk): the passes leave
// through two u32 staging buffers and bulk copies (bulk_flush_emit_pass),
// so the stores drain while the next votes run; else (k_fill_scan) the
// threads store each pass to M_H themselves (flush_emit_pass).
template <bool BULK>
__device__ __forceinline__ void fill_scan_body(const Geom &g, const Work &w, const FillCfg &c, const ScanArgs &a)
{
    extern __shared__ uint4 sm4[];
    // layout: ScanSmem (256 B) | K entries | tile | [BULK: 2 staging buffers] | HC staged hits |
    //         candidate lists (keys, votes, sorted keys, sorted votes)
    ScanSmem &ss = *reinterpret_cast<ScanSmem *>(sm4);
    uint4 *pbuf = sm4 + 16;
    uint32_t *tile = reinterpret_cast<uint32_t *>(pbuf + a.K);
    uint32_t *stg = tile + c.tile_words;
    float2 *hs = reinterpret_cast<float2 *>(stg + (BULK ? staging_words(c, g.nb) : 0u));
    uint32_t *lists = reinterpret_cast<uint32_t *>(hs + c.HC);
    __shared__ uint32_t s_hot[2], s_nc;

    const uint32_t tid = threadIdx.x, bd = blockDim.x, nb = g.nb;
    for (uint32_t k = tid; k < c.tile_words / 4; k += bd)
        sm4[16 + a.K + k] = make_uint4(0u, 0u, 0u, 0u);
    grid_dep_wait();   // the unit lists of k_scatter
    const uint32_t cta = blockIdx.x;
    ChunkList inner = interior_list(a, cta);

    __shared__ unsigned long long s_rng[2];
    __shared__ uint32_t s_dyn;
    const uint64_t items = (uint64_t)w.nu * c.strips, first = (uint64_t)w.u0 * c.strips;
    const uint64_t n_dyn = c.dyn ? dyn_items(items, gridDim.x) : 0, n_static = items - n_dyn;
    uint64_t it0, it1;
    cta_items(g, w, c, cta, gridDim.x, n_static, it0, it1, s_rng);
    uint64_t cached_es = ~0ull;
    uint32_t cached_n = 0;
    uint32_t buf_n = 0, nseq = 0, total = 0;
    uint32_t bsel = 0;   // BULK: the staging buffer of the next half pass

    auto do_item = [&](const ItemCursor &cur) {
        const uint32_t k = cur.k;
        const uint64_t es = cur.es;
        const uint32_t s = cur.s;
        const uint32_t e = cur.e;
        const uint32_t l0 = __ldg(&w.slice_off[es]), l1 = __ldg(&w.slice_off[es + 1]);   // the unit's hits
        const uint32_t i0 = k * c.W;
        const uint32_t rows = min(c.W, g.na - i0);
        const bool u16 = (l1 - l0) < 65536u;
        const uint32_t rpass = u16 ? c.W : c.W / 2;
        const uint32_t pitch = u16 ? c.pitch16 : c.pitch32;
        const uint32_t slice_lin0 = s * g.na * nb;
        const uint32_t *Ms = w.M + (size_t)e * w.n_cells + slice_lin0;
        uint32_t *Mrow = w.M + (size_t)e * w.n_cells + ((size_t)s * g.na + i0) * g.nb;
        const uint32_t r = tid % rpass, hl = tid / rpass, hstride = bd / rpass;

        for (uint32_t p0 = 0; p0 < rows; p0 += rpass) {
            const uint32_t pr = min(rpass, rows - p0);
            const uint32_t iA = i0 + p0;
            // ---- vote (no barrier first: the previous pass, the previous item's
            // hand-out or the set-up ended with one) ---------------------------
            const uint32_t i = iA + r;
            vote_pass<BlockGroup, false>(g, w, tile, hs, c.HC, es, l0, l1, cached_es, cached_n, u16, r, pr,
                                                i, hl, hstride, pitch);
            // ---- write the pass, clear the tile, emit its candidates --------
            if (BULK) {
                if (u16)
                    bulk_flush_emit_pass<true>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, tile, pitch,
                                               Mrow + (size_t)p0 * nb, pr, iA, slice_lin0, e, stg, c.W / 2, bsel,
                                               lists, s_hot, &s_nc);
                else
                    bulk_flush_emit_pass<false>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, tile, pitch,
                                                Mrow + (size_t)p0 * nb, pr, iA, slice_lin0, e, stg, c.W / 2, bsel,
                                                lists, s_hot, &s_nc);
            } else if (u16) {
                flush_emit_pass<BlockGroup, true>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, tile, pitch,
                                                  Mrow + (size_t)p0 * nb, pr, iA, slice_lin0, e, Ms, lists, s_hot,
                                                  &s_nc, nullptr);
            } else {
                flush_emit_pass<BlockGroup, false>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, tile, pitch,
                                                   Mrow + (size_t)p0 * nb, pr, iA, slice_lin0, e, Ms, lists, s_hot,
                                                   &s_nc, nullptr);
            }
        }
    };
    ItemCursor cur(g, c, first + it0);
    for (uint64_t item = it0; item < it1; ++item, cur.next(g, c))
        do_item(cur);
    finish_candidates<BlockGroup>(w, a, ss, pbuf, buf_n, nseq, total, inner, cta);
    if (c.dyn) {
        // handed-out items, each with its own list of chunks
        for (uint32_t d; (d = next_dyn_item(w, (uint32_t)n_dyn, &s_dyn)) < n_dyn;) {
            const uint32_t list = gridDim.x + d;
            inner = interior_list(a, list);
            buf_n = nseq = total = 0;
            do_item(ItemCursor(g, c, first + n_static + d));
            finish_candidates<BlockGroup>(w, a, ss, pbuf, buf_n, nseq, total, inner, list);
        }
    }
    if (BULK && threadIdx.x == 0)
        bulk_wait<0>();   // the last copies have written M_H (and read the staging) before the CTA ends
}

__global__ void __launch_bounds__(1024) k_fill_scan(Geom g, Work w, FillCfg c, ScanArgs a)
{
    fill_scan_body<false>(g, w, c, a);
}

__global__ void __launch_bounds__(1024) k_fill_bulk(Geom g, Work w, FillCfg c, ScanArgs a)
{
    fill_scan_body<true>(g, w, c, a);
}

// ---------------------------------------------------------------------------
// k_fill_ws: the fused fill with warp specialisation, one CTA per SM.
//
// 1024 threads in two groups of 16 warps: the vote group stages hits and
// votes strip passes into one of two shared-memory tiles while the flush
// group writes the other tile to M_H, clears it and emits its candidates
// (exactly as k_fill_scan does).  Tiles change hands through mbarriers --
// FULL[b] (512 vote arrivals: tile b holds a pass) and EMPTY[b] (512 flush
// arrivals: tile b is clear again) -- with bounded waits, so the votes of
// pass p + 1 run while pass p streams to HBM.  Each group keeps to its own
// named barrier; a wait that gives up makes its whole group leave (decided
// by a group-wide vote) after flagging ST_WAIT_TIMEOUT, and the other
// group's waits then give up too.
// ---------------------------------------------------------------------------
using VoteGroup = WarpGroup<1, 0, 512>;
using FlushGroup = WarpGroup<2, 512, 512>;

// Geometry of one (event, slice, strip) work item.
struct ItemInfo {
    uint64_t es;
    uint32_t s, e, l0, l1, i0, rows, rpass, pitch;   // l0, l1: the unit's hit list
    bool u16;
};

__device__ __forceinline__ ItemInfo item_info(const Geom &g, const Work &w, const FillCfg &c, const ItemCursor &cur)
{
    ItemInfo t;
    const uint32_t k = cur.k;
    t.es = cur.es;
    t.s = cur.s;
    t.e = cur.e;
    t.l0 = __ldg(&w.slice_off[t.es]);
    t.l1 = __ldg(&w.slice_off[t.es + 1]);
    t.i0 = k * c.W;
    t.rows = min(c.W, g.na - t.i0);
    t.u16 = (t.l1 - t.l0) < 65536u;
    t.rpass = t.u16 ? c.W : c.W / 2;
    t.pitch = t.u16 ? c.pitch16 : c.pitch32;
    return t;
}

__global__ void __launch_bounds__(1024, 1) k_fill_ws(Geom g, Work w, FillCfg c, ScanArgs a)
{
    extern __shared__ uint4 sm4[];
    // layout: ScanSmem (256 B) | K entries | 2 tiles | HC staged vote lines |
    //         candidate lists | 4 mbarriers (FULL 0, FULL 1, EMPTY 0, EMPTY 1)
    ScanSmem &ss = *reinterpret_cast<ScanSmem *>(sm4);
    uint4 *pbuf = sm4 + 16;
    uint32_t *tiles = reinterpret_cast<uint32_t *>(pbuf + a.K);
    float2 *hs = reinterpret_cast<float2 *>(tiles + 2 * (size_t)c.tile_words);
    uint32_t *lists = reinterpret_cast<uint32_t *>(hs + c.HC);
    uint64_t *bars = reinterpret_cast<uint64_t *>(lists + 4 * kFusedCand);
    __shared__ uint32_t s_hot[2], s_nc;

    const uint32_t tid = threadIdx.x, nb = g.nb;
    for (uint32_t k = tid; k < c.tile_words / 2; k += blockDim.x)
        reinterpret_cast<uint4 *>(tiles)[k] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        for (uint32_t q = 0; q < 4; ++q)
            mbar_init(&bars[q], VoteGroup::size());
        fence_mbar_init();
    }
    __syncthreads();   // the last block-wide barrier: the groups part here
    grid_dep_wait();   // the unit lists of k_scatter

    const uint32_t cta = blockIdx.x;
    __shared__ unsigned long long s_rng[2][2];

    if (tid < VoteGroup::size()) {
        // ---------------- vote group ----------------
        const uint32_t vr = VoteGroup::rank();
        uint64_t it0, it1;
        cta_items<VoteGroup>(g, w, c, cta, gridDim.x, (uint64_t)w.nu * c.strips, it0, it1, s_rng[0]);
        uint64_t cached_es = ~0ull;
        uint32_t cached_n = 0, p = 0;
        ItemCursor cur(g, c, (uint64_t)w.u0 * c.strips + it0);
        for (uint64_t item = it0; item < it1; ++item, cur.next(g, c)) {
            const ItemInfo t = item_info(g, w, c, cur);
            const uint32_t r = vr % t.rpass, hl = vr / t.rpass, hstride = VoteGroup::size() / t.rpass;
            for (uint32_t p0 = 0; p0 < t.rows; p0 += t.rpass, ++p) {
                const uint32_t pr = min(t.rpass, t.rows - p0);
                const uint32_t b = p & 1u;
                uint32_t *tile = tiles + (size_t)b * c.tile_words;
                if (p >= 2) {
                    const bool ok = mbar_wait_bounded(&bars[2 + b], ((p >> 1) - 1u) & 1u);
                    if (VoteGroup::sync_or(!ok)) {
                        if (vr == 0)
                            atomicOr(w.status, (uint32_t)ST_WAIT_TIMEOUT);
                        return;
                    }
                }
                const uint32_t i = t.i0 + p0 + r;
                vote_pass<VoteGroup, false>(g, w, tile, hs, c.HC, t.es, t.l0, t.l1, cached_es, cached_n,
                                                   t.u16, r, pr, i, hl, hstride, t.pitch);
                mbar_arrive(&bars[b]);   // tile b holds pass p
            }
        }
        return;
    }

    // ---------------- flush + emit group ----------------
    const uint32_t fr = FlushGroup::rank();
    uint64_t it0, it1;
    cta_items<FlushGroup>(g, w, c, cta, gridDim.x, (uint64_t)w.nu * c.strips, it0, it1, s_rng[1]);
    const ChunkList inner = interior_list(a, cta);
    uint32_t buf_n = 0, nseq = 0, total = 0, p = 0;
    bool alive = true;
    ItemCursor cur(g, c, (uint64_t)w.u0 * c.strips + it0);
    for (uint64_t item = it0; item < it1 && alive; ++item, cur.next(g, c)) {
        const ItemInfo t = item_info(g, w, c, cur);
        const uint32_t slice_lin0 = t.s * g.na * nb;
        const uint32_t *Ms = w.M + (size_t)t.e * w.n_cells + slice_lin0;
        uint32_t *Mrow = w.M + (size_t)t.e * w.n_cells + ((size_t)t.s * g.na + t.i0) * nb;
        for (uint32_t p0 = 0; p0 < t.rows; p0 += t.rpass, ++p) {
            const uint32_t pr = min(t.rpass, t.rows - p0);
            const uint32_t b = p & 1u;
            uint32_t *tile = tiles + (size_t)b * c.tile_words;
            const bool ok = mbar_wait_bounded(&bars[b], (p >> 1) & 1u);
            if (FlushGroup::sync_or(!ok)) {
                if (fr == 0)
                    atomicOr(w.status, (uint32_t)ST_WAIT_TIMEOUT);
                alive = false;
                break;
            }
            if (t.u16)
                flush_emit_pass<FlushGroup, true>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, tile, t.pitch,
                                                  Mrow + (size_t)p0 * nb, pr, t.i0 + p0, slice_lin0, t.e, Ms, lists,
                                                  s_hot, &s_nc, &bars[2 + b]);
            else
                flush_emit_pass<FlushGroup, false>(g, w, a, ss, pbuf, buf_n, nseq, total, inner, tile, t.pitch,
                                                   Mrow + (size_t)p0 * nb, pr, t.i0 + p0, slice_lin0, t.e, Ms, lists,
                                                   s_hot, &s_nc, &bars[2 + b]);
        }
    }
    finish_candidates<FlushGroup>(w, a, ss, pbuf, buf_n, nseq, total, inner, cta);
    (void)fr;
}

// ---------------------------------------------------------------------------
// k_peaks: after a fused fill (same grid), each CTA tests its candidate
// entries against their neighbours in the now complete M_H and compacts
// every chunk in place to its peaks (order kept), counting them per event.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_peaks(Geom g, Work w, ScanArgs a)
{
    grid_dep_wait();
    __shared__ uint32_t s_wsum[40];
    const uint32_t tid = threadIdx.x, bd = blockDim.x, cta = blockIdx.x;
    const uint32_t warp = tid >> 5, lane = tid & 31u, nw = (bd + 31) >> 5;
    const uint32_t nseq = a.cta_nseq[cta], sl = g.na * g.nb;
    uint32_t total = 0;
    for (uint32_t q = 0; q < nseq; ++q) {
        uint2 *dp = &a.desc[(size_t)cta * a.seq_max + q];
        const uint2 d = *dp;
        uint32_t kept = 0;
        for (uint32_t base = 0; base < d.y; base += bd) {
            const uint32_t k = base + tid;
            uint32_t has = 0;
            uint4 en = make_uint4(0u, 0u, 0u, 0u);
            if (k < d.y && d.x + k < a.entries_cap) {
                en = a.entries[d.x + k];
                const uint32_t s = en.x / sl, rem = en.x - s * sl, i = rem / g.nb, j = rem - i * g.nb;
                const uint32_t *row = w.M + (size_t)en.y * w.n_cells + (size_t)(s * g.na + i) * g.nb;
                has = is_peak_l2(row, i > 0 ? row - g.nb : nullptr, i + 1 < g.na ? row + g.nb : nullptr, j, g.nb,
                                 en.z) ? 1u : 0u;
            }
            // stable compaction: every read of this round happens before the
            // barrier, every write after, and no write passes its own read
            const uint32_t incl = warp_incl_scan(has);
            if (lane == 31u)
                s_wsum[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                const uint32_t v = lane < nw ? s_wsum[lane] : 0u;
                const uint32_t vi = warp_incl_scan(v);
                s_wsum[lane] = vi - v;
                if (lane == 31u)
                    s_wsum[32] = vi;
            }
            __syncthreads();
            if (has) {
                a.entries[d.x + kept + s_wsum[warp] + incl - 1] = en;
                atomicAdd(&a.ev_count[en.y], 1u);
            }
            kept += s_wsum[32];
            __syncthreads();
        }
        if (tid == 0)
            dp->y = kept;
        total += kept;
    }
    if (tid == 0)
        a.cta_total[cta] = total;
}

// Ascending bitonic sort of n <= kCand words in shared memory (block-wide).
__device__ void sort_u32(uint32_t *s, uint32_t n)
{
    if (n < 2)
        return;
    uint32_t P = 1;
    while (P < n)
        P <<= 1;
    for (uint32_t i = n + threadIdx.x; i < P; i += blockDim.x)
        s[i] = 0xffffffffu;
    __syncthreads();
    for (uint32_t k = 2; k <= P; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) {
                const uint32_t l = i ^ j;
                if (l > i) {
                    const uint32_t x = s[i], y = s[l];
                    if ((x > y) == ((i & k) == 0)) {
                        s[i] = y;
                        s[l] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// Test sorted candidate cells (run-local indices from global row g0) against
// their neighbours in M_H and append the peaks in order.
__device__ void test_candidates(const Geom &g, const Work &w, const ScanArgs &a, ScanSmem &ss, uint4 *pbuf,
                                uint32_t &buf_n, uint32_t &nseq, uint32_t &total, uint64_t g0,
                                const uint32_t *cand, uint32_t n)
{
    const uint32_t tid = threadIdx.x, bd = blockDim.x, nb = g.nb;
    const uint64_t rows_ev = (uint64_t)g.n_slices * g.na;
    for (uint32_t base = 0; base < n; base += bd) {
        const uint32_t k = base + tid;
        uint32_t has = 0;
        uint4 ent = make_uint4(0u, 0u, 0u, 0u);
        if (k < n) {
            const uint32_t idx = cand[k];
            const uint64_t gr = g0 + idx / nb;
            const uint32_t j = idx % nb;
            const uint32_t i = (uint32_t)(gr % g.na);
            const uint64_t row_all = gr + (uint64_t)w.u0 * g.na;   // of all matrices' rows
            const uint32_t ev = (uint32_t)(row_all / rows_ev);
            const uint32_t *row = w.M + gr * nb;
            const uint32_t v = row[j];
            if (is_peak(row, i > 0 ? row - nb : nullptr, i + 1 < g.na ? row + nb : nullptr, j, nb, v)) {
                has = 1;
                ent = make_uint4((uint32_t)((row_all - (uint64_t)ev * rows_ev) * nb) + j, ev, v, 0u);
            }
        }
        if (__syncthreads_or(has)) {
            if (buf_n + bd > a.K)
                flush_chunk(a, ss, pbuf, buf_n, nseq, interior_list(a, blockIdx.x), w.status);
            compact_entry(ss, pbuf, buf_n, has, ent, a.ev_count);
            total += ss.round_total;
        }
    }
}

// Register-streaming scan (n_b % 4 == 0): many resident warps per SM, each
// thread keeps kLdgUPT independent 16-byte streaming loads in flight; a chunk
// of a.R rows (kLdgUPT 16-byte units per thread) costs one block vote.

__global__ void __launch_bounds__(256) k_scan_ldg(Geom g, Work w, ScanArgs a)
{
    grid_dep_wait();
    extern __shared__ uint4 sm4[];
    ScanSmem &ss = *reinterpret_cast<ScanSmem *>(sm4);
    uint4 *pbuf = sm4 + 16;
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    const uint32_t nb = g.nb, nb4 = nb >> 2, T = g.threshold;
    const uint64_t G = (uint64_t)g.na * w.nu;
    const uint64_t g0 = G * blockIdx.x / gridDim.x, g1 = G * (blockIdx.x + 1) / gridDim.x;
    const uint32_t RC = a.R;
    uint32_t buf_n = 0, nseq = 0, total = 0;
    // pass 1: stream the run with no block barrier; collect the cells >= T
    // (run-local index) in a shared list, and mark their chunks (RC rows) in
    // a shared bitmap for when the list overflows
    uint32_t *hot = reinterpret_cast<uint32_t *>(pbuf + a.K);
    uint32_t *cand = hot + a.hot_words;
    __shared__ uint32_t s_ncand;
    const uint64_t n_chunks = (g1 - g0 + RC - 1) / RC;
    for (uint32_t k = tid; k < (n_chunks + 31) / 32; k += bd)
        hot[k] = 0u;
    if (tid == 0)
        s_ncand = 0u;
    __syncthreads();
    const uint4 *run = reinterpret_cast<const uint4 *>(w.M + g0 * nb);
    const uint64_t n4 = (g1 - g0) * nb4, per_chunk = (uint64_t)RC * nb4;
    for (uint64_t u0 = 0; u0 < n4; u0 += (uint64_t)kLdgUPT * bd) {
        uint4 v[kLdgUPT];
#pragma unroll
        for (uint32_t q = 0; q < kLdgUPT; ++q) {
            const uint64_t u = u0 + (uint64_t)q * bd + tid;
            v[q] = u < n4 ? __ldcs(run + u) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (uint32_t q = 0; q < kLdgUPT; ++q)
            if (max(max(v[q].x, v[q].y), max(v[q].z, v[q].w)) >= T) {
                const uint64_t u = u0 + (uint64_t)q * bd + tid;
                const uint64_t c = u / per_chunk;
                atomicOr(&hot[c >> 5], 1u << (c & 31u));
                const uint32_t vv[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
                for (uint32_t m = 0; m < 4; ++m)
                    if (vv[m] >= T) {
                        const uint32_t p = atomicAdd(&s_ncand, 1u);
                        if (p < kCand)
                            cand[p] = (uint32_t)(4 * u + m);
                    }
            }
    }
    __syncthreads();
    const uint32_t n_cand = s_ncand;
    if (n_cand <= kCand && (g1 - g0) * nb < (1ull << 32)) {
        // pass 2: the candidates in linear order, tested one per thread
        sort_u32(cand, n_cand);
        test_candidates(g, w, a, ss, pbuf, buf_n, nseq, total, g0, cand, n_cand);
    } else {
        // too many: detailed pass over the marked chunks
        for (uint64_t c = 0; c < n_chunks; ++c) {
            if (!((hot[c >> 5] >> (c & 31u)) & 1u))
                continue;
            const uint64_t ra = g0 + c * RC, rb = min(ra + RC, g1);
            scan_rows_slow<4>(g, w, a, ss, pbuf, buf_n, nseq, total, ra, rb, w.M, 0);
        }
    }
    flush_chunk(a, ss, pbuf, buf_n, nseq, interior_list(a, blockIdx.x), w.status);
    if (tid == 0) {
        a.cta_nseq[blockIdx.x] = min(nseq, a.seq_max);
        a.cta_total[blockIdx.x] = total;
    }
}

// ---------------------------------------------------------------------------
// k_order: one warp per list of chunks (a scan CTA's or a fused-fill list),
// eight lists per CTA; a list's rank is the peak total of the lists before it.
// ---------------------------------------------------------------------------
// The 32-byte output record of entry {lin within event, event, votes, .}.
__device__ __forceinline__ Peak peak_record(const Geom &g, const uint4 &en)
{
    const uint32_t lin = en.x;
    const uint32_t s = lin / (g.na * g.nb);
    const uint32_t rem = lin - s * (g.na * g.nb);
    const uint32_t i = rem / g.nb, j = rem - i * g.nb;
    Peak pk;
    pk.itheta = s / g.np;
    pk.iphi = s - pk.itheta * g.np;
    pk.ia = i;
    pk.ib = j;
    pk.votes = en.z;
    pk.a_c = a_centre(g, i);
    pk.b_c = b_centre(g, j);
    pk.event = en.y;
    return pk;
}

__global__ void __launch_bounds__(256) k_order(Geom g, Work w, ScanArgs a, OrderArgs o)
{
    grid_dep_wait();
    extern __shared__ uint32_t smo[];
    uint32_t *ev_base = smo;                  // n_events + 1
    uint32_t *red = ev_base + w.n_events + 1; // 40
    __shared__ uint32_t s_tot[32], s_last;
    const uint32_t tid = threadIdx.x, bd = blockDim.x, warp = tid >> 5, lane = tid & 31u, nw = bd >> 5;
    if (blockIdx.x == 0 && tid == 0 && o.status_out)
        *o.status_out = *w.status;   // this kernel raises nothing itself
    // one list per warp: lists c0 .. c0 + nw - 1
    const uint32_t c0 = blockIdx.x * nw, c = c0 + warp;
    const bool valid = c < a.grid;
    const uint32_t nseq = valid ? a.cta_nseq[c] : 0u, mine = valid ? a.cta_total[c] : 0u;
    const uint2 d0 = nseq ? a.desc[(size_t)c * a.seq_max] : make_uint2(0u, 0u);
    // one event or one list over all events: the rank within the event is the
    // global rank (no per-event bases)
    const bool global_rank = o.compact || w.n_events == 1;
    if (lane == 0)
        s_tot[warp] = mine;
    const bool any = __syncthreads_or(mine != 0);   // a CTA whose lists hold no peaks writes nothing

    // rank of the CTA's first list: the totals of the lists before it
    uint32_t part = 0;
    if (any)
        for (uint32_t q0 = 0; q0 < c0; q0 += 4 * bd) {   // four loads per thread in flight
            uint32_t v[4];
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) {
                const uint32_t q = q0 + k * bd + tid;
                v[k] = q < c0 ? a.cta_total[q] : 0u;
            }
            part += (v[0] + v[1]) + (v[2] + v[3]);
        }
    part = warp_incl_scan(part);
    if (lane == 31u)
        red[warp] = part;
    if (any && !global_rank)
        for (uint32_t e = tid; e < w.n_events; e += bd)
            ev_base[e] = o.ev_count[e];
    __syncthreads();
    uint32_t P = 0;
    for (uint32_t q = 0; q < nw; ++q)
        P += red[q];
    for (uint32_t q = 0; q < warp; ++q)   // the CTA's lists before this warp's
        P += s_tot[q];
    __syncthreads();
    if (any && !global_rank)
        block_exclusive_scan(ev_base, w.n_events, red);

    for (uint32_t q = 0; q < (mine ? nseq : 0u); ++q) {
        const uint2 d = q == 0 ? d0 : a.desc[(size_t)c * a.seq_max + q];
        for (uint32_t k = lane; k < d.y; k += 32u) {
            if (d.x + k >= a.entries_cap)
                break;
            const uint4 en = a.entries[d.x + k];
            const uint32_t e = en.y;
            const uint32_t pos = global_rank ? P + k : P + k - ev_base[e];
            if (pos < o.capacity)
                o.out[o.compact ? (size_t)pos : (size_t)e * o.capacity + pos] = peak_record(g, en);
        }
        P += d.y;
    }
    if (global_rank) {
        // no other CTA reads the per-event counts: the first one publishes and
        // resets them (and the entry counter), and no CTA waits for the others
        if (blockIdx.x == 0) {
            for (uint32_t e = tid; e < w.n_events; e += bd) {
                o.counts[e] = o.ev_count[e];
                o.ev_count[e] = 0u;
            }
            if (tid == 0)
                *o.g_count = 0u;
        }
        return;
    }
    if (blockIdx.x == 0)
        for (uint32_t e = tid; e < w.n_events; e += bd)
            o.counts[e] = o.ev_count[e];

    // Every CTA read the per-event counts: the last CTA to finish resets the
    // counters for the next scan.
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(o.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (uint32_t e = tid; e < w.n_events; e += bd)
            o.ev_count[e] = 0u;
        if (tid == 0) {
            *o.g_count = 0u;
            *o.ticket = 0u;
        }
    }
}

// ---------------------------------------------------------------------------
// k_fill_tma: the fill fused with the peaks, one warp per tile.
//
// A pass is W A-rows of one (event, slice) unit.  A warp votes it into a u32
// shared-memory tile of its own, laid out as M_H's rows, sends the tile to
// M_H as one bulk copy (cp.async.bulk, shared -> global), finds the pass's
// peaks in it while the copy reads, and clears it for its next pass.  Nothing
// a warp does waits for another warp: the latencies of one pass (offsets,
// lines, votes, copy) overlap with the other warps' passes.
//
// Order of the passes: a CTA's warps take a pass each of its runs (run i of
// CTA c is run i * grid + c: c.run = warps neighbouring passes), and the last
// passes go to whichever warp of the grid comes first, so that the whole grid
// writes one neighbourhood of M_H at any time (compressible memory wants that)
// and the hits' uneven spread over the slices averages out.
//
// The peaks are found where the votes are: a vote that lifts its cell from
// T - 1 to T lists the cell, and the listed cells are compared with their
// neighbours in the tile.  For a cell on the first or last row of the pass
// the votes of the row beyond are counted from the unit's lines (nothing waits
// for the warp that owns it), or k_edges compares them later.  Each pass leaves
// {first entry, count} in pass_peaks, in pass order, for k_order_passes.
//
// Where slices may be so crowded that their passes outlast the rest (TEAM, chosen
// by the host), passes above a share of the votes wait until a CTA's warps have no
// other pass, and then take all of them (team_passes).
//
// Bound: writing M_H where votes are few (paper event, one launch: 42 us for
// 268 MB, 54 MB of which reach HBM, as M_H is compressed; upgrade event, in
// flight: 498 us for 4.3 GB), the votes' instructions where they are many
// (admission windows, 38 M candidate votes: 76 us).  Against CTAs of 512
// threads that shared a tile, with three block barriers per pass and the peak
// tests in a kernel of their own (events with three contexts in flight, with
// what else changed around it): paper event 50.0 -> 33.7 us, windows 142.5 ->
// 63.9 us, batch of 100 events 4424 -> 3090 us, four sectors 73.3 -> 33.8 us.
// Tried on the way: the old tile
// rotation behind a feeding warp, 48 us in flight (one barrier per pass, every
// pass's latency exposed), and voting, draining and feeding warps around four
// tiles, 44-47 us (the hand-overs cost more than the votes).
// ---------------------------------------------------------------------------

// Cells of a pass that reached T: keys r * n_b + j, the first kTileCand.
struct PassList {
    uint32_t n;
    uint32_t cand[kTileCand];
};

// A pass: the unit's nc hits (lines and records), and its rows.
struct TilePass {
    const float2 *lines;
    const float4 *recs;
    uint32_t nc, iA, pr;
};

// A line that is no vote in any row (for lanes without a hit).
__device__ __forceinline__ float2 no_line() { return make_float2(1.0e9f, 0.0f); }

// The first 32 * kAhead of n lines, lane by lane.
__device__ __forceinline__ void first_lines(float2 (&l)[kAhead], const float2 *lines, uint32_t n)
{
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (uint32_t k = 0; k < kAhead; ++k)
        l[k] = 32u * k + lane < n ? __ldg(lines + 32u * k + lane) : no_line();
}

// 1 + the bins of the votes of line l (record *rec) in the R A bins from i on
// (x: those bins less g.mid); 0 or above n_b for none.  on: this lane has a
// hit.  As vote_bin_line, the R of them side by side and the rule behind one
// branch.
template <int R>
__device__ __forceinline__ void line_bins(const Geom &g, const float2 l, const float (&x)[R], uint32_t i,
                                          const float4 *rec, bool on, uint32_t (&j1)[R])
{
    const float big = 12582912.0f;
    const float lim = __fmaf_rn(-g.err_v, fabsf(l.y), g.err_half);
    const uint32_t near = lim > 0.0f ? g.nb + 1u : ~0u;   // bins whose edges matter
    bool ask = false;
    float d[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const float t = __fmaf_rn(l.y, x[q], l.x);
        const float k = __fadd_rn(t, big);
        d[q] = __fsub_rn(t, __fsub_rn(k, big));
        j1[q] = __float_as_uint(k) - (__float_as_uint(big) - 1u);
        ask |= !(fabsf(d[q]) <= lim) && j1[q] <= near;
    }
    if (ask && on) {
        const float4 h = __ldg(rec);
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (!(fabsf(d[q]) <= lim) && j1[q] <= near)
                j1[q] = 1u + (uint32_t)vote_bin(g, __fmul_rn(2.0f, a_centre(g, i + q)), h.x, h.y, h.z);
    }
}

// Who works on a pass: a warp (the rule), or all warps of the CTA (team_passes).
struct WarpCrew {
    static __device__ __forceinline__ uint32_t rank() { return threadIdx.x & 31u; }
    static __device__ __forceinline__ uint32_t size() { return 32u; }
    static __device__ __forceinline__ uint32_t warp() { return 0u; }
    static __device__ __forceinline__ uint32_t warps() { return 1u; }
    static __device__ __forceinline__ void sync() { __syncwarp(); }
};
struct CtaCrew {
    static __device__ __forceinline__ uint32_t rank() { return threadIdx.x; }
    static __device__ __forceinline__ uint32_t size() { return blockDim.x; }
    static __device__ __forceinline__ uint32_t warp() { return threadIdx.x >> 5; }
    static __device__ __forceinline__ uint32_t warps() { return blockDim.x >> 5; }
    static __device__ __forceinline__ void sync() { __syncthreads(); }
};

// The first 32 * kAhead lines of this warp's share of a pass's n: groups of 32 *
// kAhead go to the crew's warps in turn.
template <class C>
__device__ __forceinline__ void crew_lines(float2 (&l)[kAhead], const float2 *lines, uint32_t n)
{
    const uint32_t h = C::warp() * 32u * kAhead;
    first_lines(l, lines + h, n > h ? n - h : 0u);
}

// The votes of a pass into its tile (l: crew_lines; the next
// ones are loaded that far ahead): R rows at a time, a lane holds one hit's
// line; consecutive lanes hold consecutive hits, whose B columns, and so whose
// banks, differ.  A vote that lifts its cell from T - 1 to T lists the cell.
// The R atomics are issued unconditionally, a lane without a vote adding 0 to
// a word of its own (spare): behind a branch each would wait for the one
// before it (102 cycles per atomic and warp, against 21 so).  AGG:
// warp-aggregated increments -- the lanes voting for the same cell find each
// other (match.any) and their lowest lane adds their number with one atomic;
// the cell is listed by the add that takes it from below T to T or more.
template <bool AGG, int R, class C>
__device__ __forceinline__ void vote_tile(const Geom &g, uint32_t *tile, const TilePass &P, float2 (&l)[kAhead],
                                          PassList &L, uint32_t spare)
{
    const uint32_t nb = g.nb, T = g.threshold, lane = threadIdx.x & 31u;
    for (uint32_t r0 = 0; r0 < P.pr; r0 += R) {
        if (r0)
            crew_lines<C>(l, P.lines, P.nc);
        float x[R];
        uint32_t row[R], most[R];   // per row: its first cell, less 1; the largest bin, plus 1 (0 beyond the pass)
#pragma unroll
        for (int q = 0; q < R; ++q) {
            x[q] = __int2float_rn((int)(P.iA + r0 + q) - g.mid);
            row[q] = (r0 + q) * nb - 1u;
            most[q] = r0 + q < P.pr ? nb : 0u;
        }
        // 32 hits, one per lane
        auto vote = [&](const float2 line, uint32_t h) {
            uint32_t j1[R], at[R], n[R], old[R], top = 0;
            line_bins<R>(g, line, x, P.iA + r0, P.recs + h, h < P.nc, j1);
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const bool ok = j1[q] - 1u < most[q];
                at[q] = ok ? row[q] + j1[q] : spare;
                n[q] = ok ? 1u : 0u;
            }
            if (AGG) {
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const uint32_t peers = __match_any_sync(0xffffffffu, at[q]);
                    n[q] = lane == (uint32_t)(__ffs(peers) - 1) ? n[q] * (uint32_t)__popc(peers) : 0u;
                }
            }
#pragma unroll
            for (int q = 0; q < R; ++q)
                old[q] = atomicAdd(&tile[at[q]], n[q]);
#pragma unroll
            for (int q = 0; q < R; ++q)
                top = max(top, old[q] + n[q]);
            if (top >= T) {
#pragma unroll
                for (int q = 0; q < R; ++q)
                    if (old[q] < T && old[q] + n[q] >= T) {
                        const uint32_t p = atomicAdd(&L.n, 1u);
                        if (p < kTileCand)
                            L.cand[p] = at[q];
                    }
            }
        };
        const uint32_t step = C::warps() * 32u * kAhead;
        for (uint32_t h0 = C::warp() * 32u * kAhead; h0 < P.nc; h0 += step) {
            float2 ahead[kAhead];
            const uint32_t h1 = h0 + step;
            first_lines(ahead, P.lines + h1, P.nc > h1 ? P.nc - h1 : 0u);
#pragma unroll
            for (uint32_t k = 0; k < kAhead; ++k) {
                if (h0 + 32u * k < P.nc)
                    vote(l[k], h0 + 32u * k + lane);
                l[k] = ahead[k];
            }
        }
    }
}

// The votes of A row i into row[0 .. n_b).  AHEAD: with kAhead lines per thread
// loaded ahead (for units of many hits).
template <class C, bool AHEAD>
__device__ __forceinline__ void vote_row(const Geom &g, uint32_t *row, const TilePass &P, uint32_t i)
{
    C::sync();
    if (!AHEAD) {
        for (uint32_t h = C::rank(); h < P.nc; h += C::size()) {
            const uint32_t j = vote_bin_line(g, __ldg(P.lines + h), i, P.recs + h);
            if (j < g.nb)
                atomicAdd(&row[j], 1u);
        }
        C::sync();
        return;
    }
    const uint32_t step = C::size() * kAhead;
    auto load = [&](float2 (&l)[kAhead], uint32_t h0) {
#pragma unroll
        for (uint32_t k = 0; k < kAhead; ++k)
            l[k] = h0 + k * C::size() < P.nc ? __ldg(P.lines + h0 + k * C::size()) : no_line();
    };
    float2 l[kAhead];
    load(l, C::rank());
    for (uint32_t h0 = C::rank(); h0 < P.nc; h0 += step) {
        float2 ahead[kAhead];
        load(ahead, h0 + step);
#pragma unroll
        for (uint32_t k = 0; k < kAhead; ++k) {
            const uint32_t h = h0 + k * C::size();
            const uint32_t j = vote_bin_line(g, l[k], i, P.recs + h, h < P.nc);
            if (j < g.nb)
                atomicAdd(&row[j], 1u);
            l[k] = ahead[k];
        }
    }
    C::sync();
}

// The votes of the rows before (above) and behind (below) a pass into row[0 .. n_b)
// and row[n_b .. 2 n_b).
template <class C>
__device__ __forceinline__ void vote_rows_beyond(const Geom &g, uint32_t *row, const TilePass &P, bool above, bool below)
{
    const uint32_t step = C::size() * kAhead, nb = g.nb;
    const float x[2] = {__int2float_rn((int)P.iA - 1 - g.mid), __int2float_rn((int)(P.iA + P.pr) - g.mid)};
    auto load = [&](float2 (&l)[kAhead], uint32_t h0) {
#pragma unroll
        for (uint32_t k = 0; k < kAhead; ++k)
            l[k] = h0 + k * C::size() < P.nc ? __ldg(P.lines + h0 + k * C::size()) : no_line();
    };
    float2 l[kAhead];
    load(l, C::rank());
    for (uint32_t h0 = C::rank(); h0 < P.nc; h0 += step) {
        float2 ahead[kAhead];
        load(ahead, h0 + step);
#pragma unroll
        for (uint32_t k = 0; k < kAhead; ++k) {
            const uint32_t h = h0 + k * C::size();
            const float x0[1] = {x[0]}, x1[1] = {x[1]};
            uint32_t j0[1], j1[1];
            line_bins<1>(g, l[k], x0, P.iA - 1u, P.recs + h, above && h < P.nc, j0);
            line_bins<1>(g, l[k], x1, P.iA + P.pr, P.recs + h, below && h < P.nc, j1);
            if (above && j0[0] - 1u < nb)
                atomicAdd(&row[j0[0] - 1u], 1u);
            if (below && j1[0] - 1u < nb)
                atomicAdd(&row[nb + j1[0] - 1u], 1u);
            l[k] = ahead[k];
        }
    }
    C::sync();
}

// Where a pass's peaks go: the pass and segment counts, and the entries.
struct PassOut {
    uint32_t e, lin0;   // event, linear index of the pass's first cell
    uint32_t pass;
    // room for n entries; a warp calls it
    __device__ __forceinline__ uint32_t claim(const Work &w, const ScanArgs &a, uint32_t n) const
    {
        uint32_t base = 0;
        if ((threadIdx.x & 31u) == 0) {
            if (n) {
                base = atomicAdd(a.g_count, n);
                atomicAdd(&w.seg_peaks[pass >> w.seg_shift], n);
                atomicAdd(&a.ev_count[e], n);
                if (base + n > a.entries_cap || base + n < base)
                    atomicOr(w.status, (uint32_t)ST_SCRATCH_OVERFLOW);
            }
            w.pass_peaks[pass] = make_uint2(base, n);
        }
        return __shfl_sync(0xffffffffu, base, 0);
    }
    __device__ __forceinline__ void put(const ScanArgs &a, uint32_t at, uint32_t key, uint32_t v) const
    {
        if (at < a.entries_cap)
            a.entries[at] = make_uint4(lin0 + key, e, v, 0u);
    }
};

// The test of cell `key` of a tile of pr rows against its neighbours in the tile.
__device__ __forceinline__ bool peak_in_tile(const uint32_t *tile, uint32_t pr, uint32_t nb, uint32_t key, uint32_t v)
{
    const uint32_t r = key / nb, j = key - r * nb;
    const uint32_t *row = tile + r * nb;
    return is_peak(row, r > 0 ? row - nb : nullptr, r + 1 < pr ? row + nb : nullptr, j, nb, v);
}

// Many peaks: the cells that are peaks, a bit each (cleared), go out in order.
// One warp calls it.
__device__ __forceinline__ void put_bits(const Work &w, const ScanArgs &a, const PassOut &O, const uint32_t *tile,
                                         uint32_t *bits, uint32_t words)
{
    const uint32_t lane = threadIdx.x & 31u, full = 0xffffffffu;
    __syncwarp();
    uint32_t n = 0;
    for (uint32_t q = lane; q < words; q += 32u)
        n += (uint32_t)__popc(bits[q]);
    uint32_t base = O.claim(w, a, __reduce_add_sync(full, n));
    for (uint32_t q0 = 0; q0 < words; q0 += 32u) {
        const uint32_t q = q0 + lane;
        uint32_t m = q < words ? bits[q] : 0u;
        if (q < words)
            bits[q] = 0u;
        const uint32_t c = (uint32_t)__popc(m), incl = warp_incl_scan(c);
        for (uint32_t at = base + incl - c; m; m &= m - 1u, ++at) {
            const uint32_t key = 32u * q + (uint32_t)(__ffs(m) - 1);
            O.put(a, at, key, tile[key]);
        }
        base += __shfl_sync(full, incl, 31);
    }
    __syncwarp();
}

// The peaks of a pass by a look at every cell of its tile (bits: one bit per cell,
// zero between calls).  above, below: the pass has a row before, behind it that
// its first, last row is compared with: that row is voted into a row of the tile
// which the test does not need (the tile holds at least two), and that row is
// voted anew after it; with rows to spare (scratch: two rows, zero between calls)
// both are voted there, in one go.  reading: a bulk copy of the crew's first
// thread may still read the tile.
template <class C, bool AHEAD>
__device__ __forceinline__ void search_cells(const Geom &g, const Work &w, const ScanArgs &a, const TilePass &P,
                                             const PassOut &O, uint32_t *tile, uint32_t *bits, bool above, bool below,
                                             bool reading, uint32_t *scratch)
{
    const uint32_t lane = threadIdx.x & 31u, nb = g.nb, pr = P.pr, last = (pr - 1u) * nb;
    const uint32_t cells = pr * nb, words = (cells + 31u) / 32u;
    for (uint32_t q = C::warp(); q < words; q += C::warps()) {
        const uint32_t key = 32u * q + lane;
        const uint32_t v = key < cells ? tile[key] : 0u;
        const uint32_t m = __ballot_sync(0xffffffffu, v >= g.threshold && peak_in_tile(tile, pr, nb, key, v));
        if (lane == 0)
            bits[q] = m;
    }
    if ((above || below) && !scratch && reading && C::rank() == 0)
        bulk_wait_read<0>();
    C::sync();
    // drop the peaks of a row (its first cell: key0) that the row beyond outdoes
    auto compare = [&](const uint32_t *row, uint32_t key0, bool before) {
        for (uint32_t j = C::rank(); j < nb; j += C::size()) {
            const uint32_t key = key0 + j, b = 1u << (key & 31u);
            const uint32_t most = max(row[j], max(j ? row[j - 1] : 0u, j + 1 < nb ? row[j + 1] : 0u));
            if ((bits[key >> 5] & b) && !(before ? tile[key] > most : tile[key] >= most))
                atomicAnd(&bits[key >> 5], ~b);
        }
    };
    if (scratch) {
        if (above || below) {
            vote_rows_beyond<C>(g, scratch, P, above, below);
            if (above)
                compare(scratch, 0u, true);
            if (below)
                compare(scratch + nb, last, false);
            C::sync();
            for (uint32_t j = C::rank(); j < 2u * nb; j += C::size())
                scratch[j] = 0u;
        }
        if (C::warp() == 0)
            put_bits(w, a, O, tile, bits, words);
        C::sync();
        return;
    }
    auto beyond = [&](uint32_t i, uint32_t key0, uint32_t spare, bool before) {
        uint32_t *row = tile + spare * nb;
        auto clear = [&]() {
            C::sync();
            for (uint32_t j = C::rank(); j < nb; j += C::size())
                row[j] = 0u;
        };
        clear();
        vote_row<C, AHEAD>(g, row, P, i);
        compare(row, key0, before);
        clear();
        if (spare < pr)
            vote_row<C, AHEAD>(g, row, P, P.iA + spare);
        C::sync();
    };
    if (above)
        beyond(P.iA - 1u, 0u, 1u, true);
    if (below)
        beyond(P.iA + pr, last, pr > 1u ? 0u : 1u, false);
    if (C::warp() == 0)
        put_bits(w, a, O, tile, bits, words);
    C::sync();
}

// The peaks of a warp's pass (its own tile and list; bits as search_cells).
// reading: a bulk copy may still read the tile.  edges_later: the rows beyond the
// pass are left to k_edges.  MANY: units may hold many hits.  Every lane calls it.
template <bool MANY>
__device__ __forceinline__ void pass_search(const Geom &g, const Work &w, const ScanArgs &a, const TilePass &P,
                                            const PassOut &O, uint32_t *tile, const PassList &L, uint32_t *bits,
                                            bool reading, bool edges_later)
{
    const uint32_t lane = threadIdx.x & 31u, nb = g.nb, n_c = L.n, full = 0xffffffffu, pr = P.pr;
    const uint32_t last = (pr - 1u) * nb;
    const uint32_t cells = pr * nb, words = (cells + 31u) / 32u;
    // the pass has a row of the slice before / behind it, which this kernel compares with
    const bool above = !edges_later && P.iA > 0, below = !edges_later && P.iA + pr < g.na;
    bool list = n_c <= kTileCand;
    if (MANY && list && P.nc > kListHits && (above || below)) {
        // many hits: counting them for every listed cell of the first and last row
        // against voting the rows beyond and looking at every cell
        uint32_t edge = 0;
        for (uint32_t k = lane; k < n_c; k += 32u)
            edge += (above && L.cand[k] < nb) + (below && L.cand[k] >= last);
        edge = __reduce_add_sync(full, edge);
        list = (uint64_t)edge * P.nc <= 8u * P.nc + 64u * words;
    }
    if (!list) {
        search_cells<WarpCrew, MANY>(g, w, a, P, O, tile, bits, above, below, reading, nullptr);
        return;
    }
    // one listed cell per lane;
    // the three cells of row i next to the cells j of the lanes in m, counted
    // hit by hit: the most votes one of them holds, for each lane in m
    auto beyond = [&](uint32_t m, uint32_t i, uint32_t j) {
        uint32_t c0 = 0, c1 = 0, c2 = 0;
        const float x[1] = {__int2float_rn((int)i - g.mid)};
        float2 l = lane < P.nc ? __ldg(P.lines + lane) : no_line();
        for (uint32_t h0 = 0; h0 < P.nc; h0 += 32u) {
            const uint32_t h = h0 + lane;
            uint32_t b[1];
            line_bins<1>(g, l, x, i, P.recs + h, h < P.nc, b);
            const uint32_t j1 = b[0] - 1u < nb ? b[0] : 0x80000000u;   // no cell is next to that
            l = h + 32u < P.nc ? __ldg(P.lines + h + 32u) : no_line();
            for (uint32_t k = m; k; k &= k - 1u) {
                const uint32_t src = (uint32_t)(__ffs(k) - 1);
                const uint32_t d = j1 - __shfl_sync(full, j, src);
                const uint32_t b0 = __ballot_sync(full, d == 0u), b1 = __ballot_sync(full, d == 1u),
                               b2 = __ballot_sync(full, d == 2u);
                if (lane == src) {
                    c0 += (uint32_t)__popc(b0);
                    c1 += (uint32_t)__popc(b1);
                    c2 += (uint32_t)__popc(b2);
                }
            }
        }
        return max(c1, max(c0, c2));
    };
    for (uint32_t k0 = 0; k0 < n_c; k0 += 32u) {
        const bool has = k0 + lane < n_c;
        const uint32_t key = has ? L.cand[k0 + lane] : ~0u;
        const uint32_t v = has ? tile[key] : 0u;
        bool keep = has && peak_in_tile(tile, pr, nb, key, v);
        uint32_t m = __ballot_sync(full, keep && above && key < nb);
        if (m) {
            const uint32_t most = beyond(m, P.iA - 1u, key);
            if ((m >> lane) & 1u)
                keep = v > most;
        }
        m = __ballot_sync(full, keep && below && key >= last);
        if (m) {
            const uint32_t most = beyond(m, P.iA + pr, key - last);
            if ((m >> lane) & 1u)
                keep = v >= most;
        }
        if (n_c > 32u) {
            if (keep)
                atomicOr(&bits[key >> 5], 1u << (key & 31u));
            continue;
        }
        m = __ballot_sync(full, keep);
        uint32_t rank = 0;
        const uint32_t n = (uint32_t)__popc(m);
        for (; m; m &= m - 1u)
            rank += __shfl_sync(full, key, __ffs(m) - 1) < key;
        const uint32_t base = O.claim(w, a, n);
        if (keep)
            O.put(a, base + rank, key, v);
    }
    if (n_c > 32u)
        put_bits(w, a, O, tile, bits, words);
}

// A finished tile to M_H: whole 16 bytes as one bulk copy, which the crew's first
// thread issues, up to three words on either side by hand.
template <class C>
__device__ __forceinline__ void send_tile(uint32_t *dst, const uint32_t *tile, uint64_t cell0, uint32_t cells)
{
    const uint32_t head = min((uint32_t)(-cell0 & 3u), cells), mid = (cells - head) & ~3u, rank = C::rank();
    if (rank == 0) {
        if (mid)
            bulk_store_evict_first(dst + head, tile + head, mid * 4u);
        bulk_commit();
    }
    if (rank < cells - mid) {
        const uint32_t k = rank < head ? rank : mid + rank;
        dst[k] = tile[k];
    }
}

// Pass `pass` of unit `unit`, whose hits are the list entries off.x .. off.y.
__device__ __forceinline__ TilePass tile_pass(const Geom &g, const Work &w, const TileCfg &c, uint32_t pass,
                                              uint32_t unit, uint2 off)
{
    TilePass P;
    P.iA = (pass - unit * c.strips) * c.W;
    P.pr = min(c.W, g.na - P.iA);
    P.lines = w.lines + off.x;
    P.recs = w.list + off.x;
    P.nc = off.y - off.x;
    return P;
}

__device__ __forceinline__ PassOut pass_out(const Geom &g, const TilePass &P, uint32_t pass, uint32_t unit)
{
    const uint32_t e = unit / g.n_slices;
    return PassOut{e, ((unit - e * g.n_slices) * g.na + P.iA) * g.nb, pass};
}

// Passes of units with more hits than this are left to whole CTAs (team_passes):
// such a pass is more than the fair share of one of the grid's warps, so the
// others would end long before it.
__device__ __forceinline__ uint32_t team_limit(const Geom &g, const Work &w, const TileCfg &c)
{
    const uint64_t total = __ldcg(&w.slice_off[w.n_events * g.n_slices]);
    const uint64_t share = total * c.strips / (c.team_share * gridDim.x);
    return (uint32_t)min(max(share, (uint64_t)kTeamHits), (uint64_t)0xffffffffu);
}

// The passes of units with more than `limit` hits, each by all warps of a CTA in
// the first warp's tile: the votes, and the look at every cell, are dealt out to
// the warps.  The passes are numbered over those units in order and handed out by
// a counter.  Out of line: most launches have none.
//
// Crowded slices are bound by one warp's chain of votes, and by its look at the
// rows beyond the pass, unless they are dealt out so (us per event, one warp per
// pass / this): 16384 hits in one slice of 128 x 4096 bins, threshold 3, 620 / 73,
// peaks only, threshold 10, 4568 / 67; 4 slices of 16 x 1024 bins with 4096 hits each,
// threshold 3, 161 / 43; 64 slices of 128 x 4096 bins with 4096 hits each, peaks only,
// threshold 10, 3508 / 381.
template <bool STORE>
__device__ __noinline__ void team_passes(const Geom &g, const Work &w, const TileCfg &c, const ScanArgs &a,
                                         uint32_t limit, uint32_t *tile0, uint32_t spare0, uint32_t *s_word)
{
    const uint32_t nb = g.nb, tid = threadIdx.x, U = w.n_events * g.n_slices;
    uint32_t *bits = tile0 + c.tile_words;
    PassList &L = *reinterpret_cast<PassList *>(bits + tile_bit_words(c.tile_words));
    uint32_t *scratch = c.warps > 1u ? tile0 + tile_warp_words(c.tile_words) : nullptr;   // the second warp's tile
    auto claim = [&]() {
        __syncthreads();   // the last claim is read, the tile clear
        if (tid == 0)
            *s_word = atomicAdd(&w.ctr[CTR_TEAM], 1u);
        __syncthreads();
        return *s_word;
    };
    auto vote_pass = [&](uint32_t unit, uint32_t strip) {
        const uint32_t pass = unit * c.strips + strip;
        const TilePass P = tile_pass(g, w, c, pass, unit,
                                     make_uint2(__ldcg(&w.slice_off[unit]), __ldcg(&w.slice_off[unit + 1u])));
        const uint64_t cell0 = (uint64_t)unit * ((uint64_t)g.na * nb) + (uint64_t)P.iA * nb;
        const uint32_t shift = (uint32_t)(cell0 & 3u);
        uint32_t *tile = tile0 + shift;
        float2 l[kAhead];
        crew_lines<CtaCrew>(l, P.lines, P.nc);
        if (P.pr > 2u)
            vote_tile<false, 4, CtaCrew>(g, tile, P, l, L, spare0 - shift);
        else
            vote_tile<false, 2, CtaCrew>(g, tile, P, l, L, spare0 - shift);
        if (STORE)
            fence_proxy_async_smem();
        __syncthreads();
        if (STORE)
            send_tile<CtaCrew>(w.M + cell0, tile, cell0, P.pr * nb);
        const bool here = !(STORE && c.edges_later);   // the rows beyond are compared here
        if (L.n)
            search_cells<CtaCrew, true>(g, w, a, P, pass_out(g, P, pass, unit), tile, bits, here && P.iA > 0,
                                        here && P.iA + P.pr < g.na, STORE, scratch);
        else if (tid == 0)
            w.pass_peaks[pass] = make_uint2(0u, 0u);
        if (STORE && tid == 0)
            bulk_wait_read<0>();
        __syncthreads();
        if (tid == 0)
            L.n = 0u;
        for (uint32_t q = tid; q < c.tile_words / 4u; q += blockDim.x)
            reinterpret_cast<uint4 *>(tile0)[q] = make_uint4(0u, 0u, 0u, 0u);
    };
    auto crowded = [&](uint32_t u) {
        return u < U && __ldcg(&w.slice_off[u + 1u]) - __ldcg(&w.slice_off[u]) > limit;
    };
    uint32_t mine = ~0u, before = 0;   // the claimed pass; the passes of the crowded units so far
    for (uint32_t u0 = 0; u0 < U; u0 += 32u) {
        if (u0 % blockDim.x == 0) {   // a block's width of units at once: mostly none is crowded
            if (!__syncthreads_or(crowded(u0 + tid))) {
                u0 += blockDim.x - 32u;
                continue;
            }
            if (mine == ~0u)
                mine = claim();
        }
        uint32_t m = __ballot_sync(0xffffffffu, crowded(u0 + (tid & 31u)));
        for (; m; m &= m - 1u, before += c.strips)
            for (; mine - before < c.strips; mine = claim())
                vote_pass(u0 + (uint32_t)(__ffs(m) - 1), mine - before);
    }
    if (STORE && tid == 0)
        bulk_wait<0>();
}

// STORE: the tiles go to M_H, else the peaks are all that is wanted (the same
// passes without the copies: 29.6 us for a paper event, 20.0 us per event in
// flight; the u16 tiles of 512 threads that it replaces, whose cross-pass tests
// went through rows in global memory and k_peaks, 31.8 and 31.5 us).  AGG:
// warp-aggregated vote increments (vote_tile).  passes: over all events; runs:
// runs of c.run passes per CTA, the passes behind them being handed out.
template <bool STORE, bool AGG, bool TEAM>
__global__ void __launch_bounds__(kTileWarps * 32, 2) k_fill_tma(const __grid_constant__ Geom g,
                                                              const __grid_constant__ Work w,
                                                              const __grid_constant__ TileCfg c,
                                                              const __grid_constant__ ScanArgs a, uint32_t passes,
                                                              uint32_t runs)
{
    extern __shared__ uint4 sm4[];
    // layout: per tile warp a tile, its bits, its list and 32 idle words.  (TEAM: warps
    // beyond those only take part in team_passes.)
    __shared__ uint32_t s_word;   // warps with passes to come; TEAM: team_passes' claim
    const uint32_t nb = g.nb, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t warps = TEAM ? c.warps : blockDim.x >> 5;
    const uint32_t mine = tile_warp_words(c.tile_words);
    uint32_t *tile0 = reinterpret_cast<uint32_t *>(sm4) + (TEAM ? warp % warps : warp) * mine;
    uint32_t *bits = tile0 + c.tile_words;
    PassList &L = *reinterpret_cast<PassList *>(bits + tile_bit_words(c.tile_words));
    const uint32_t *idle = reinterpret_cast<uint32_t *>(&L) + tile_list_words() + lane;   // the lane's own word
    if (!TEAM || warp < warps)
        for (uint32_t k = lane; k < mine / 4u; k += 32u)
            reinterpret_cast<uint4 *>(tile0)[k] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0)
        s_word = warps;
    __syncthreads();
    grid_dep_wait();   // the unit lists

    // The warp's passes: one of each of the CTA's runs, then the ones handed out
    // (the first is the warp's own number in the grid).  Lane 0 claims a
    // handed-out pass one pass before its number is needed.
    const uint32_t fixed = runs * c.run * gridDim.x;
    uint32_t turn = 0, claimed = blockIdx.x * warps + warp;
    auto next_pass = [&]() {
        if (turn < runs)
            return (turn++ * gridDim.x + blockIdx.x) * c.run + warp;
        const uint32_t q = __shfl_sync(0xffffffffu, claimed, 0);
        if (q >= passes - fixed)
            return passes;
        if (lane == 0)
            claimed = warps * gridDim.x + atomicAdd(&w.ctr[CTR_DYN], 1u);
        return fixed + q;
    };
    auto offsets = [&](uint32_t pass) {
        if (pass >= passes)
            return make_uint2(0u, 0u);
        const uint32_t u = pass / c.strips;
        return make_uint2(__ldcg(&w.slice_off[u]), __ldcg(&w.slice_off[u + 1]));
    };
    // The next pass's lines are loaded while this one's tile leaves, and the
    // offsets of the one behind it: nothing that a pass begins with is waited for.
    const bool idler = TEAM && warp >= warps;
    uint32_t pass = idler ? passes : next_pass(), next = idler ? passes : next_pass();
    uint2 off = offsets(pass), next_off = offsets(next);
    const uint32_t limit = TEAM ? team_limit(g, w, c) : 0u;
    float2 l[kAhead];
    first_lines(l, w.lines + off.x, off.y - off.x);
    while (pass < passes) {
        const uint32_t unit = pass / c.strips;
        const TilePass P = tile_pass(g, w, c, pass, unit, off);
        const bool team = TEAM && P.nc > limit;   // left to team_passes
        // the pass's first cell lies in the tile as in M_H: at the same address modulo 16 bytes
        const uint64_t cell0 = (uint64_t)unit * ((uint64_t)g.na * nb) + (uint64_t)P.iA * nb;
        uint32_t *tile = tile0 + (uint32_t)(cell0 & 3u);
        if (!team) {
            const uint32_t spare = (uint32_t)(idle - tile);
            if (P.pr > 2u)
                vote_tile<AGG, 4, WarpCrew>(g, tile, P, l, L, spare);
            else
                vote_tile<AGG, 2, WarpCrew>(g, tile, P, l, L, spare);
            if (STORE)
                fence_proxy_async_smem();   // this lane's counts, visible to the copy engine
            __syncwarp();
            // ---- the pass leaves
            if (STORE)
                send_tile<WarpCrew>(w.M + cell0, tile, cell0, P.pr * nb);
        }
        first_lines(l, w.lines + next_off.x, next_off.y - next_off.x);
        const uint32_t next2 = next_pass();
        const uint2 next2_off = offsets(next2);
        if (!team) {
            // ---- its peaks
            if (L.n)
                pass_search<TEAM>(g, w, a, P, pass_out(g, P, pass, unit), tile, L, bits, STORE, STORE && c.edges_later);
            else if (lane == 0)
                w.pass_peaks[pass] = make_uint2(0u, 0u);
            // ---- the tile is cleared once the copy has read it
            if (STORE && lane == 0)
                bulk_wait_read<0>();
            __syncwarp();
            if (lane == 0)
                L.n = 0u;
#pragma unroll 8
            for (uint32_t k = lane; k < c.tile_words / 4u; k += 32u)
                reinterpret_cast<uint4 *>(tile0)[k] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
        }
        pass = next;
        off = next_off;
        next = next2;
        next_off = next2_off;
    }
    if (STORE && lane == 0)
        bulk_wait<0>();   // the warp's copies have written M_H (and read its tile) before the CTA ends
    if (TEAM) {
        __syncthreads();
        team_passes<STORE>(g, w, c, a, limit, reinterpret_cast<uint32_t *>(sm4),
                           (uint32_t)(idle - reinterpret_cast<uint32_t *>(sm4)), &s_word);
    }
    if (TEAM ? tid == 0 : lane == 0 && atomicSub(&s_word, 1u) == 1u) {
        __threadfence();
        if (atomicAdd(&w.ctr[CTR_DYN_DONE], 1u) == gridDim.x - 1) {   // nobody claims any more
            w.ctr[CTR_DYN] = 0u;
            w.ctr[CTR_DYN_DONE] = 0u;
            if (TEAM)
                w.ctr[CTR_TEAM] = 0u;
        }
    }
}

// ---------------------------------------------------------------------------
// k_fill_add: accumulating fills of few hits.  A warp takes kAddRows A rows of
// one (event, slice) unit and adds its votes to M_H one by one (reductions in
// L2, results unused): a fill that touches few cells does not read and write
// the others, as k_fill_priv does.  Bound by the L2's reductions and by the
// sectors of M_H that they bring in.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_fill_add(Geom g, Work w, uint32_t strips)
{
    grid_dep_wait();   // the unit lists
    const uint32_t lane = threadIdx.x & 31u, nb = g.nb;
    const uint64_t slice_cells = (uint64_t)g.na * nb, items = (uint64_t)w.n_events * g.n_slices * strips;
    const uint64_t stride = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t it = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < items; it += stride) {
        const uint32_t u = (uint32_t)(it / strips), i0 = (uint32_t)(it - (uint64_t)u * strips) * kAddRows;
        const uint32_t i1 = min(i0 + kAddRows, g.na), l0 = w.slice_off[u], nc = w.slice_off[u + 1] - l0;
        uint32_t *Ms = w.M + (uint64_t)u * slice_cells;   // unit u = e * n_slices + s, n_cells = n_slices * slice_cells
        for (uint32_t h = lane; h < nc; h += 32u) {
            const float2 l = __ldg(w.lines + l0 + h);
            const float4 *rec = w.list + l0 + h;
            for (uint32_t i = i0; i < i1; i += 4u) {
                float x[4];
                uint32_t j1[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    x[q] = __int2float_rn((int)(i + q) - g.mid);
                line_bins<4>(g, l, x, i, rec, true, j1);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (j1[q] - 1u < nb && i + q < i1)
                        atomicAdd(Ms + (size_t)(i + q) * nb + (j1[q] - 1u), 1u);
            }
        }
    }
}

// The peaks (or candidates) of a segment of 1 << seg_shift passes, as k_edges and
// k_order_passes read them, one thread per pass: each pass's first rank in the
// segment and first entry.  Returns how many there are.
constexpr uint32_t kNoPeak = 0xffffffffu;
struct SegmentPeaks {
    uint32_t off[kOrderPasses], base[kOrderPasses], wsum[kOrderPasses / 32];
};

__device__ __forceinline__ uint32_t load_segment(SegmentPeaks &sp, const Work &w, uint32_t seg, uint64_t passes)
{
    const uint32_t tid = threadIdx.x, warp = tid >> 5;
    const uint64_t pass = ((uint64_t)seg << w.seg_shift) + tid;
    const uint2 d = pass < passes && tid >> w.seg_shift == 0u ? w.pass_peaks[pass] : make_uint2(0u, 0u);
    const uint32_t incl = warp_incl_scan(d.y);
    if ((tid & 31u) == 31u)
        sp.wsum[warp] = incl;
    __syncthreads();
    uint32_t off = incl - d.y, n = 0;
    for (uint32_t q = 0; q < kOrderPasses / 32; ++q) {
        off += q < warp ? sp.wsum[q] : 0u;
        n += sp.wsum[q];
    }
    sp.off[tid] = off;
    sp.base[tid] = d.x;
    __syncthreads();
    return n;
}

// The pass (of the segment) that holds the segment's peak k: the last one that
// starts at or before k.
__device__ __forceinline__ uint32_t segment_pass(const SegmentPeaks &sp, uint32_t k)
{
    uint32_t lo = 0, hi = kOrderPasses - 1;
    while (lo < hi) {
        const uint32_t m = (lo + hi + 1) >> 1;
        if (sp.off[m] <= k)
            lo = m;
        else
            hi = m - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// k_edges: the comparisons that the tile fill left (TileCfg::edges_later).  An
// entry on the first or last row of its pass is compared with the row beyond in
// M_H; .w becomes the rank in the segment plus 1, or kNoPeak (0, as the fill
// leaves it: the position is the rank), and the segment's and events' counts
// become those of the peaks.  Voting the row beyond anew, as passes of few hits
// do, costs a pass its hits over again for both of its edges; here a comparison
// is three words out of L2.  One event in flight and alone, without and with
// this: admission windows 87.0 -> 63.9 and 143.7 -> 96.5 us, 24000 hits in the
// paper's matrix 79.5 -> 58.9 and 138 -> 98.6 us.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kOrderPasses) k_edges(Geom g, Work w, TileCfg c, ScanArgs a, uint64_t passes)
{
    grid_dep_wait();
    __shared__ SegmentPeaks sp;
    __shared__ uint32_t s_kept[kOrderPasses / 32];
    const uint32_t tid = threadIdx.x, seg = blockIdx.x, warp = tid >> 5, lane = tid & 31u, nb = g.nb, full = 0xffffffffu;
    if (w.seg_peaks[seg] == 0u)
        return;
    const uint32_t n = load_segment(sp, w, seg, passes);
    uint32_t kept = 0;
    for (uint32_t k0 = 0; k0 < n; k0 += kOrderPasses) {
        const uint32_t k = k0 + tid;
        bool has = k < n, keep = has;
        uint32_t at = 0, e = 0;
        if (has) {
            const uint32_t q = segment_pass(sp, k);
            at = sp.base[q] + (k - sp.off[q]);
            has = keep = at < a.entries_cap;
            if (has) {
                const uint4 en = a.entries[at];
                e = en.y;
                const uint64_t pass = ((uint64_t)seg << w.seg_shift) + q;
                const uint32_t unit = (uint32_t)(pass / c.strips), strip = (uint32_t)(pass - (uint64_t)unit * c.strips);
                const uint32_t first = strip * c.W, last = min(first + c.W, g.na) - 1u;
                const uint32_t row = en.x / nb, j = en.x - row * nb, i = row % g.na;
                // the most votes of the three cells of row i next to column j
                auto beyond = [&](uint32_t i) {
                    const uint32_t *r = w.M + ((uint64_t)unit * g.na + i) * nb + j;
                    return max(__ldcg(r), max(j ? __ldcg(r - 1) : 0u, j + 1u < nb ? __ldcg(r + 1) : 0u));
                };
                if (i == first && i > 0u)
                    keep = en.z > beyond(i - 1u);
                if (keep && i == last && i + 1u < g.na)
                    keep = en.z >= beyond(i + 1u);
            }
        }
        const uint32_t m = __ballot_sync(full, keep);
        if (lane == 0)
            s_kept[warp] = (uint32_t)__popc(m);
        __syncthreads();
        uint32_t rank = kept + (uint32_t)__popc(m & ((1u << lane) - 1u));
        for (uint32_t q = 0; q < kOrderPasses / 32; ++q) {
            rank += q < warp ? s_kept[q] : 0u;
            kept += s_kept[q];
        }
        if (has)
            a.entries[at].w = keep ? rank + 1u : kNoPeak;
        for (uint32_t out = __ballot_sync(full, has && !keep); out;) {   // by event
            const uint32_t src = (uint32_t)(__ffs(out) - 1), es = __shfl_sync(full, e, src);
            const uint32_t same = __ballot_sync(full, e == es) & out;
            if (lane == src)
                atomicSub(&a.ev_count[es], (uint32_t)__popc(same));
            out &= ~same;
        }
        __syncthreads();
    }
    if (tid == 0)
        w.seg_peaks[seg] = kept;
}

// ---------------------------------------------------------------------------
// k_order_passes: the peaks of k_fill_tma's passes into one list, ascending.
// A CTA takes a segment of 1 << seg_shift passes: its first rank is the sum of
// the segments before it, and one thread per peak finds its pass by a search
// over the segment's prefix sums.  (One event, or one list over all events.)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kOrderPasses) k_order_passes(Geom g, Work w, ScanArgs a, OrderArgs o,
                                                               uint64_t passes)
{
    grid_dep_wait();
    __shared__ SegmentPeaks sp;
    __shared__ uint32_t s_before[kOrderPasses / 32];
    const uint32_t tid = threadIdx.x, seg = blockIdx.x;
    const uint32_t mine = w.seg_peaks[seg];
    if (seg == 0) {
        if (tid == 0 && o.status_out)
            *o.status_out = *w.status;
        // no other CTA reads the counters: this one leaves them as k_order does
        for (uint32_t e = tid; e < w.n_events; e += kOrderPasses) {
            o.counts[e] = o.ev_count[e];
            o.ev_count[e] = 0u;
        }
        if (tid == 0)
            *o.g_count = 0u;
    }
    if (mine == 0)
        return;
    uint32_t before = 0;
    for (uint32_t q = tid; q < seg; q += kOrderPasses)
        before += w.seg_peaks[q];
    before = __reduce_add_sync(0xffffffffu, before);
    if ((tid & 31u) == 0)
        s_before[tid >> 5] = before;
    const uint32_t n = load_segment(sp, w, seg, passes);
    uint32_t rank0 = 0;
    for (uint32_t q = 0; q < kOrderPasses / 32; ++q)
        rank0 += s_before[q];
    for (uint32_t k = tid; k < n; k += kOrderPasses) {
        const uint32_t q = segment_pass(sp, k), at = sp.base[q] + (k - sp.off[q]);
        if (at >= a.entries_cap)
            continue;
        const uint4 en = a.entries[at];
        const uint32_t rank = en.w ? en.w - 1u : k;
        if (en.w != kNoPeak && (uint64_t)rank0 + rank < o.capacity)
            o.out[rank0 + rank] = peak_record(g, en);
    }
}

} // namespace htk

// ---------------------------------------------------------------------------
// Launchers (host).
// ---------------------------------------------------------------------------
namespace htk {

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) only when a launch needs
// more than was already allowed for the kernel on this device: the attribute
// call is a driver round trip that would otherwise cost every launch.
static cudaError_t allow_smem(const void *kernel, size_t bytes)
{
    constexpr int kSlots = 16, kDevs = 64;
    static std::atomic<const void *> keys[kSlots];
    static std::atomic<int> allowed[kSlots][kDevs];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs)
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    int slot = -1;
    for (int i = 0; i < kSlots && slot < 0; ++i) {
        const void *k = keys[i].load(std::memory_order_acquire);
        if (k == kernel)
            slot = i;
        else if (!k) {
            const void *expect = nullptr;
            if (keys[i].compare_exchange_strong(expect, kernel) || expect == kernel)
                slot = i;
        }
    }
    if (slot < 0)
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    std::atomic<int> &a = allowed[slot][dev];
    if ((int)bytes <= a.load(std::memory_order_acquire))
        return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) {
        int cur = a.load();
        while ((int)bytes > cur && !a.compare_exchange_weak(cur, (int)bytes)) {
        }
    }
    return e;
}

// Launch with programmatic stream serialisation allowed (see grid_dep_wait).
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), uint32_t grid, uint32_t block, size_t smem,
                              cudaStream_t st, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

cudaError_t launch_bin(const Geom &g, const Work &w, uint32_t grid, cudaStream_t st)
{
    const size_t smem = w.hit_off ? ((size_t)w.n_events + 1) * 4 : 0;
    if (smem > 32 * 1024) {
        cudaError_t e = allow_smem((const void *)k_bin, smem);
        if (e != cudaSuccess)
            return e;
    }
    return launch_pdl(k_bin, grid, 256, smem, st, g, w);
}

cudaError_t launch_scatter(const Geom &g, const Work &w, uint32_t grid, cudaStream_t st)
{
    return launch_pdl(k_scatter, grid, 256, 0, st, g, w);
}

size_t bin_cluster_smem_bytes(const Geom &g, uint32_t n_events)
{
    return ((size_t)3 * n_events * g.n_slices + 1 + n_events + 1) * 4;
}

bool bin_cluster_supported(size_t smem)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kBinClusterMax);
    cfg.blockDim = dim3(kBinClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kBinClusterMax;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (allow_smem((const void *)k_bin_cluster, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, (const void *)k_bin_cluster, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

cudaError_t launch_bin_cluster(const Geom &g, const Work &w, uint32_t cs, cudaStream_t st)
{
    const size_t smem = bin_cluster_smem_bytes(g, w.n_events);   // <= kBinClusterSmem, allowed by bin_cluster_supported
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(kBinClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_bin_cluster, g, w);
}

size_t fill_scan_smem_bytes(const FillCfg &c, const ScanArgs &a, uint32_t nb)
{
    return 16 * sizeof(uint4) + (size_t)a.K * sizeof(uint4) + (size_t)c.tile_words * 4 +
           (size_t)staging_words(c, nb) * 4 + (size_t)c.HC * 8 +
           (size_t)4 * kFusedCand * 4;
}

cudaError_t launch_fill_scan(const Geom &g, const Work &w, const FillCfg &c, const ScanArgs &a, uint32_t grid,
                             cudaStream_t st)
{
    const size_t smem = fill_scan_smem_bytes(c, a, g.nb);
    const void *k = c.bulk ? (const void *)k_fill_bulk : (const void *)k_fill_scan;
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess)
        return e;
    return c.bulk ? launch_pdl(k_fill_bulk, grid, c.threads, smem, st, g, w, c, a)
                  : launch_pdl(k_fill_scan, grid, c.threads, smem, st, g, w, c, a);
}

size_t fill_ws_smem_bytes(const FillCfg &c, const ScanArgs &a)
{
    return 16 * sizeof(uint4) + (size_t)a.K * sizeof(uint4) + (size_t)2 * c.tile_words * 4 + (size_t)c.HC * 8 +
           (size_t)4 * kFusedCand * 4 + 4 * sizeof(uint64_t);
}

cudaError_t launch_fill_ws(const Geom &g, const Work &w, const FillCfg &c, const ScanArgs &a, uint32_t grid,
                           cudaStream_t st)
{
    const size_t smem = fill_ws_smem_bytes(c, a);
    cudaError_t e = allow_smem((const void *)k_fill_ws, smem);
    if (e != cudaSuccess)
        return e;
    return launch_pdl(k_fill_ws, grid, kWsThreads, smem, st, g, w, c, a);
}

cudaError_t fill_ws_occupancy(const FillCfg &c, const ScanArgs &a, int *blocks_per_sm)
{
    const size_t smem = fill_ws_smem_bytes(c, a);
    cudaError_t e = allow_smem((const void *)k_fill_ws, smem);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_fill_ws, kWsThreads, smem);
}

cudaError_t launch_peaks(const Geom &g, const Work &w, const ScanArgs &a, uint32_t grid, cudaStream_t st)
{
    return launch_pdl(k_peaks, grid, 256, 0, st, g, w, a);
}

using TileKernel = void (*)(Geom, Work, TileCfg, ScanArgs, uint32_t, uint32_t);
static TileKernel tile_kernel(const TileCfg &c, bool store)
{
    if (!store)
        return c.team_share ? k_fill_tma<false, false, true> : k_fill_tma<false, false, false>;
    if (c.vote_agg)
        return c.team_share ? k_fill_tma<true, true, true> : k_fill_tma<true, true, false>;
    return c.team_share ? k_fill_tma<true, false, true> : k_fill_tma<true, false, false>;
}

cudaError_t launch_fill_tma(const Geom &g, const Work &w, const TileCfg &c, const ScanArgs &a, uint32_t grid,
                            bool store, cudaStream_t st)
{
    const size_t smem = tile_smem_bytes(c);
    const TileKernel k = tile_kernel(c, store);
    cudaError_t e = allow_smem((const void *)k, smem);
    if (e != cudaSuccess)
        return e;
    // The SMs do not write at one rate: an eighth of the passes is handed out at
    // run time (upgrade event, alone: 689 us with 3 passes per warp handed out,
    // 636 us with an eighth, 639 us with a quarter, 786 us with half of them:
    // handed-out neighbours go to different SMs, which share no lines in L1).
    const uint32_t passes = (uint32_t)tile_passes(g, c, w.n_events);
    const uint32_t handed = std::max(kHandedOut * c.warps * grid, passes / 8u);
    const uint32_t runs = passes > handed ? (passes - handed) / (grid * c.run) : 0u;
    return launch_pdl(k, grid, (c.team_share ? kTileWarps : c.warps) * 32u, smem, st, g, w, c, a, passes, runs);
}

cudaError_t fill_tma_occupancy(const TileCfg &c, bool store, int *blocks_per_sm)
{
    const size_t smem = tile_smem_bytes(c);
    const TileKernel k = tile_kernel(c, store);
    cudaError_t e = allow_smem((const void *)k, smem);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, (int)c.warps * 32, smem);
}

cudaError_t launch_order_passes(const Geom &g, const Work &w, const ScanArgs &a, const OrderArgs &o, uint64_t passes,
                                cudaStream_t st)
{
    return launch_pdl(k_order_passes, (uint32_t)(((passes - 1) >> w.seg_shift) + 1), kOrderPasses, 0, st, g, w, a, o,
                      passes);
}

cudaError_t launch_edges(const Geom &g, const Work &w, const TileCfg &c, const ScanArgs &a, uint64_t passes,
                         cudaStream_t st)
{
    return launch_pdl(k_edges, (uint32_t)(((passes - 1) >> w.seg_shift) + 1), kOrderPasses, 0, st, g, w, c, a, passes);
}

cudaError_t fill_scan_occupancy(const FillCfg &c, const ScanArgs &a, uint32_t nb, int *blocks_per_sm)
{
    const size_t smem = fill_scan_smem_bytes(c, a, nb);
    const void *k = c.bulk ? (const void *)k_fill_bulk : (const void *)k_fill_scan;
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, c.threads, smem);
}

size_t fill_smem_bytes(const FillCfg &c)
{
    return (size_t)c.tile_words * 4 + (size_t)c.HC * 8;
}

cudaError_t launch_fill_priv(const Geom &g, const Work &w, const FillCfg &c, uint32_t grid,
                             cudaStream_t st)
{
    const size_t smem = fill_smem_bytes(c);
    cudaError_t e = allow_smem((const void *)k_fill_priv, smem);
    if (e != cudaSuccess)
        return e;
    return launch_pdl(k_fill_priv, grid, c.threads, smem, st, g, w, c);
}

cudaError_t launch_fill_add(const Geom &g, const Work &w, uint32_t num_sms, cudaStream_t st)
{
    const uint32_t strips = (g.na + kAddRows - 1) / kAddRows;
    const uint64_t items = (uint64_t)w.n_events * g.n_slices * strips;
    return launch_pdl(k_fill_add, (uint32_t)std::min<uint64_t>((items + 7) / 8, num_sms * 8u), 256, 0, st, g, w, strips);
}

cudaError_t launch_copy(uint32_t *dst, const uint32_t *src, uint64_t n, cudaStream_t st)
{
    const uint64_t ctas = (n / 8u + 2u * kCopyThreads - 1) / (2u * kCopyThreads);
    return launch_pdl(k_copy, (uint32_t)std::max<uint64_t>(1, ctas), kCopyThreads, 0, st, dst, src, n);
}

cudaError_t launch_clear(uint32_t *M, uint64_t words, uint32_t grid, cudaStream_t st)
{
    return launch_pdl(k_clear, grid, 512, 0, st, M, words);
}

cudaError_t launch_fill_naive(const Geom &g, const Work &w, uint32_t num_sms, cudaStream_t st)
{
    // a block over A; as many blocks as are resident at once (2048 threads per SM)
    const uint32_t threads = g.na >= 1024 ? 1024 : ((g.na + 31) / 32) * 32;
    const size_t smem = ((size_t)g.nb + 1) * 4 <= 48u * 1024u ? ((size_t)g.nb + 1) * 4 : 0;
    return launch_pdl(k_fill_naive, num_sms * (2048 / threads), threads, smem, st, g, w);
}

size_t scan_smem_bytes(const ScanArgs &a)
{
    return 16 * sizeof(uint4) + (size_t)a.K * sizeof(uint4) + (size_t)a.S * a.slot_words * 4 +
           (size_t)a.hot_words * 4 + (a.hot_words ? (size_t)kCand * 4 : 0);
}

static const void *scan_kernel(int kind)
{
    switch (kind) {
    case SCAN_BULK:
        return (const void *)k_scan_tma;
    case SCAN_LDG:
        return (const void *)k_scan_ldg;
    default:
        return (const void *)k_scan_direct;
    }
}

cudaError_t launch_scan(const Geom &g, const Work &w, const ScanArgs &a, int kind, cudaStream_t st)
{
    const size_t smem = scan_smem_bytes(a);
    cudaError_t e = allow_smem((const void *)scan_kernel(kind), smem);
    if (e != cudaSuccess)
        return e;
    if (kind == SCAN_BULK)
        return launch_pdl(k_scan_tma, a.grid, 256, smem, st, g, w, a);
    if (kind == SCAN_LDG)
        return launch_pdl(k_scan_ldg, a.grid, 256, smem, st, g, w, a);
    return launch_pdl(k_scan_direct, a.grid, 256, smem, st, g, w, a);
}



// ---------------------------------------------------------------------------
// k_wait_probe: the failure path of the bounded waits, on demand.  One
// thread waits on a shared-memory mbarrier that nothing arrives at, giving
// up after limit_ns (at most kWaitNs) or kWaitIters polls, and flags
// ST_WAIT_TIMEOUT exactly as a real wait that gave up does.
// ---------------------------------------------------------------------------
__global__ void k_wait_probe(uint32_t *status, uint64_t limit_ns)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0)
        return;
    mbar_init(&bar, 1u);   // one arrival expected, none will come
    fence_mbar_init();
    const uint64_t t0 = global_ns();
    bool done = false;
    for (uint32_t it = 0; it < kWaitIters && !done; ++it) {
        done = mbar_try_wait(&bar, 0u);
        if ((it & 255u) == 255u && global_ns() - t0 > limit_ns)
            break;
    }
    if (!done)
        atomicOr(status, (uint32_t)ST_WAIT_TIMEOUT);
}

cudaError_t launch_wait_probe(uint32_t *status, uint32_t limit_ms, cudaStream_t st)
{
    const uint64_t ns = (uint64_t)limit_ms * 1000000ull;
    k_wait_probe<<<1, 32, 0, st>>>(status, ns < kWaitNs ? ns : kWaitNs);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// k_peaks4d: the 4-D (80-neighbour) maxima rule as a filter of the 2-D list.
//
// A cell's 8 neighbours in its own (A, B) slice are among its 80 neighbours
// in (theta, phi, A, B), so every 4-D peak is a 2-D peak: the filter takes
// the 2-D peaks (ascending linear index) and keeps those that also beat the
// up to 72 cells of the adjacent slices -- strictly the ones in an earlier
// slice (smaller linear index), with >= the ones in a later slice; phi does
// not wrap.  One warp per peak: its lanes read the 72 cells at once (three
// rounds of 32) and a warp vote decides; the keep flags go to `keep`, and
// the last CTA to finish (ticket) compacts the kept peaks in order.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_peaks4d(Geom g, const uint32_t *M, const Peak *in, const uint32_t *n_in,
                                                 uint32_t cap_in, uint8_t *keep, Peak *out, uint32_t cap_out,
                                                 uint32_t *n_out, uint32_t *ticket, uint32_t *status)
{
    __shared__ uint32_t s_warp[32], s_total, s_last;
    grid_dep_wait();   // the 2-D list of k_order
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5, nw = blockDim.x >> 5;
    const uint32_t n_all = __ldcg(n_in);
    const uint32_t n = min(n_all, cap_in);
    const int nt = (int)g.nt, np = (int)g.np, na = (int)g.na, nb = (int)g.nb;
    for (uint32_t q = blockIdx.x * nw + wid; q < n; q += gridDim.x * nw) {
        const Peak p = in[q];
        const int t = (int)p.itheta, f = (int)p.iphi, i = (int)p.ia, j = (int)p.ib;
        bool ok = true;
#pragma unroll
        for (uint32_t round = 0; round < 3; ++round) {
            const uint32_t k = lane + 32u * round;   // neighbour k: slice k / 9, cell k % 9
            if (k < 72u) {
                const uint32_t sl = k / 9u, cell = k - sl * 9u;
                const uint32_t ts = sl < 4u ? sl : sl + 1u;   // the 3 x 3 (theta, phi) offsets but (0, 0)
                const int dt = (int)(ts / 3u) - 1, df = (int)(ts % 3u) - 1;
                const int tt = t + dt, ff = f + df, ii = i + (int)(cell / 3u) - 1, jj = j + (int)(cell % 3u) - 1;
                if (tt >= 0 && tt < nt && ff >= 0 && ff < np && ii >= 0 && ii < na && jj >= 0 && jj < nb) {
                    const uint32_t w = M[(((size_t)tt * np + ff) * na + ii) * (size_t)nb + jj];
                    const bool before = dt < 0 || (dt == 0 && df < 0);
                    ok = ok && (before ? p.votes > w : p.votes >= w);
                }
            }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (lane == 0)
            keep[q] = ok ? 1u : 0u;
    }
    // the last CTA to finish compacts the kept peaks in order
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last)
        return;
    __threadfence();
    if (n_all > cap_in && tid == 0)
        atomicOr(status, (uint32_t)ST_SCRATCH_OVERFLOW);   // the 2-D list was cut: the filter would miss peaks
    uint32_t base = 0;
    for (uint32_t r0 = 0; r0 < n; r0 += blockDim.x) {
        const uint32_t q = r0 + tid;
        const bool kq = q < n && __ldcg(&keep[q]) != 0u;
        const uint32_t bal = __ballot_sync(0xffffffffu, kq);
        if (lane == 0)
            s_warp[wid] = __popc(bal);
        __syncthreads();
        if (wid == 0) {
            const uint32_t c = lane < nw ? s_warp[lane] : 0u;
            const uint32_t incl = warp_incl_scan(c);
            if (lane < nw)
                s_warp[lane] = incl - c;   // exclusive prefix of the warp totals
            if (lane == 31)
                s_total = incl;
        }
        __syncthreads();
        const uint32_t pos = base + s_warp[wid] + __popc(bal & ((1u << lane) - 1u));
        if (kq && pos < cap_out)
            out[pos] = in[q];
        base += s_total;
        __syncthreads();   // s_warp, s_total free for the next round
    }
    if (tid == 0) {
        *n_out = base;
        *ticket = 0u;
    }
}

cudaError_t launch_peaks4d(const Geom &g, const uint32_t *M, const Peak *in, const uint32_t *n_in, uint32_t cap_in,
                           uint8_t *keep, Peak *out, uint32_t cap_out, uint32_t *n_out, uint32_t *ticket,
                           uint32_t *status, uint32_t grid, cudaStream_t st)
{
    return launch_pdl(k_peaks4d, grid, 256u, (size_t)0, st, g, M, in, n_in, cap_in, keep, out, cap_out, n_out,
                      ticket, status);
}

// ---------------------------------------------------------------------------
// k_atomic_rate: the L2-atomic roofline the naive fill is measured against.
// Every thread adds 1 to per_thread words of buf picked by a linear
// congruential sequence of its own (masked to the footprint, a power of two
// words); the results are unused, so the adds are reductions performed in L2.
// ---------------------------------------------------------------------------
__global__ void k_atomic_rate(uint32_t *buf, uint32_t mask, uint32_t per_thread, uint32_t seed)
{
    uint32_t x = (blockIdx.x * blockDim.x + threadIdx.x) * 2654435761u ^ seed;
    for (uint32_t i = 0; i < per_thread; ++i) {
        x = x * 1664525u + 1013904223u;
        atomicAdd(&buf[(x >> 4) & mask], 1u);
    }
}

cudaError_t launch_atomic_rate(uint32_t *buf, uint32_t mask, uint32_t per_thread, uint32_t seed, uint32_t grid,
                               cudaStream_t st)
{
    k_atomic_rate<<<grid, 256, 0, st>>>(buf, mask, per_thread, seed);
    return cudaGetLastError();
}

cudaError_t launch_order(const Geom &g, const Work &w, const ScanArgs &a, const OrderArgs &o,
                         cudaStream_t st)
{
    const size_t smem = (w.n_events + 1 + 40) * sizeof(uint32_t);
    if (smem > 48 * 1024) {
        cudaError_t e = allow_smem((const void *)k_order, smem);
        if (e != cudaSuccess)
            return e;
    }
    // one list per warp, eight per CTA
    return launch_pdl(k_order, (a.grid + 7) / 8, 256, smem, st, g, w, a, o);
}

cudaError_t scan_occupancy(int kind, size_t smem, int *blocks_per_sm)
{
    const void *k = scan_kernel(kind);
    cudaError_t e = allow_smem((const void *)k, smem);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, 256, smem);
}

cudaError_t fill_occupancy(const FillCfg &c, int *blocks_per_sm)
{
    const size_t smem = fill_smem_bytes(c);
    cudaError_t e = allow_smem((const void *)k_fill_priv, smem);
    if (e != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_fill_priv, c.threads, smem);
}

} // namespace htk
