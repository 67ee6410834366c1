// C ABI: phi sectors (ht_sectors_*).
//
// Sec. 4 splits the transverse plane into four phi sectors, read out
// independently, runs one Hough transform per sector with a lighter matrix
// M_H(A, B, theta) and merges the results.  A sector's matrix is its phi bins
// of the unsplit M_H, and as the maxima rule compares (A, B) neighbours within
// a slice, the merged peaks are the unsplit peaks.  On one GPU the sectors are
// therefore parts of one context's matrix: one binning, one fill and one
// ordering serve them all, and the list comes out merged.  (A context, a
// stream and four launches per sector, and a merge kernel, took 54 us per
// paper-scale event in four sectors with three events in flight, where this
// takes 34 us.)
#include "ht_engine.h"
#include "ht_geom.h"
#include "ht_trace.h"

#include <cstdio>
#include <string>

namespace hte {
ht_status report(ht_status s, const std::string &msg);   // ht_api.cu
Engine &ctx_engine(ht_ctx *c);                            // ht_api.cu
} // namespace hte

struct ht_sectors {
    uint32_t S = 0, m = 0;            // sectors, phi bins per sector
    uint32_t max_hits = 0;
    ht_ctx *ctx = nullptr;            // the unsplit binning
    cudaStream_t stream = nullptr;    // the object's own stream
    // the end of the last call, and of the last one that was captured (in the
    // capture cap_id): calls run in the order they are made, on whichever streams
    cudaEvent_t done = nullptr, cap_done = nullptr;
    bool done_pending = false;
    unsigned long long done_id = 0;   // the stream's id (not its handle, which another stream may get)
    unsigned long long cap_id = 0;
    bool poisoned = false;
};

namespace {

ht_status sec_fail(ht_sectors *s, cudaError_t e, const char *what)
{
    s->poisoned = true;
    char buf[320];
    std::snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    return hte::report(HT_E_CUDA, buf);
}

#define SCK(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return sec_fail(sec, e_, #call);                                                       \
    } while (0)

ht_status check_sec(ht_sectors *sec)
{
    if (!sec)
        return hte::report(HT_E_INVAL, "sectors object is NULL");
    if (sec->poisoned)
        return hte::report(HT_E_STATE, "sectors object failed earlier (HT_E_CUDA); destroy it");
    return HT_OK;
}

// The context's answer; its message stands.
ht_status pass_on(ht_sectors *sec, ht_status s)
{
    if (s == HT_E_CUDA || s == HT_E_STATE)
        sec->poisoned = true;
    return s;
}

// Run a step of the object on st, behind the step before it whatever stream
// that took: `call` enqueues it.  A captured step and an eager one do not wait for each
// other (a capture cannot wait for work outside it, nor anything for an event
// inside it): the order of a graph's launch is its launcher's.
template <class F>
ht_status in_order(ht_sectors *sec, cudaStream_t st, F call)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    SCK(cudaStreamGetCaptureInfo(st, &cs, &id));
    const bool captured = cs != cudaStreamCaptureStatusNone;
    if (captured) {
        if (sec->cap_id == id)
            SCK(cudaStreamWaitEvent(st, sec->cap_done, 0));
    } else {
        SCK(cudaStreamGetId(st, &id));
        if (sec->done_pending && sec->done_id != id)
            SCK(cudaStreamWaitEvent(st, sec->done, 0));
    }
    const ht_status s = pass_on(sec, call());
    if (sec->poisoned)
        return s;
    SCK(cudaEventRecord(captured ? sec->cap_done : sec->done, st));
    (captured ? sec->cap_id : sec->done_id) = id;
    if (!captured)
        sec->done_pending = true;
    return s;
}

} // namespace

extern "C" {

ht_status ht_sectors_destroy(ht_sectors *sec)
{
    if (!sec)
        return HT_OK;
    if (sec->stream)
        cudaStreamSynchronize(sec->stream);
    if (sec->done_pending)
        cudaEventSynchronize(sec->done);
    ht_destroy(sec->ctx);
    if (sec->done)
        cudaEventDestroy(sec->done);
    if (sec->cap_done)
        cudaEventDestroy(sec->cap_done);
    if (sec->stream)
        cudaStreamDestroy(sec->stream);
    delete sec;
    return HT_OK;
}

ht_status ht_sectors_create(const ht_binning *binning, const ht_ranges *ranges, uint32_t threshold,
                            uint32_t n_sectors, uint32_t max_hits, ht_sectors **out)
{
    if (!out)
        return hte::report(HT_E_INVAL, "out is NULL");
    *out = nullptr;
    std::string why;
    if (!htg::validate(binning, ranges, threshold, &why))
        return hte::report(HT_E_INVAL, why);
    if (n_sectors < 1 || binning->n_phi % n_sectors)
        return hte::report(HT_E_INVAL, "n_sectors must be >= 1 and divide n_phi");
    if (binning->win_phi && n_sectors > 1)
        return hte::report(HT_E_INVAL, "phi sectors need win_phi == 0 (a window would reach the next sector)");
    if (max_hits < 1)
        return hte::report(HT_E_INVAL, "max_hits must be >= 1");
    // the sectors' phi ranges, which a caller could state for itself
    const double lo = htg::snap_quarter(ranges->phi_min), hi = htg::snap_quarter(ranges->phi_max);
    for (uint32_t k = 0; k < n_sectors; ++k)
        if (!((float)(lo + (hi - lo) * k / n_sectors) < (float)(lo + (hi - lo) * (k + 1) / n_sectors)))
            return hte::report(HT_E_INVAL, "sector phi ranges collapse in float; use fewer sectors");
    ht_sectors *sec = new (std::nothrow) ht_sectors();
    if (!sec)
        return hte::report(HT_E_NOMEM, "host allocation failed");
    sec->S = n_sectors;
    sec->m = binning->n_phi / n_sectors;
    sec->max_hits = max_hits;
    const ht_status s = ht_create(binning, ranges, threshold, max_hits, &sec->ctx);
    if (s != HT_OK) {
        const std::string msg = std::string("sector context: ") + ht_last_error();
        ht_sectors_destroy(sec);
        return hte::report(s, msg);
    }
    cudaError_t e;
    if ((e = cudaStreamCreateWithFlags(&sec->stream, cudaStreamNonBlocking)) != cudaSuccess ||
        (e = cudaEventCreateWithFlags(&sec->done, cudaEventDisableTiming)) != cudaSuccess ||
        (e = cudaEventCreateWithFlags(&sec->cap_done, cudaEventDisableTiming)) != cudaSuccess) {
        cudaGetLastError();
        ht_sectors_destroy(sec);
        return hte::report(HT_E_CUDA, std::string("sector setup: ") + cudaGetErrorString(e));
    }
    *out = sec;
    return HT_OK;
}

ht_status ht_sectors_fill(ht_sectors *sec, const float *x, const float *y, const float *z, uint32_t n_hits,
                          uint32_t flags, void *stream)
{
    hte::TraceRange tr("ht_sectors_fill");
    ht_status s = check_sec(sec);
    if (s != HT_OK)
        return s;
    if (flags & ~(uint32_t)(HT_MEM_DEVICE | HT_ACCUMULATE | HT_FILL_NAIVE | HT_PEAKS_ONLY))
        return hte::report(HT_E_INVAL, "unknown flag");
    if (n_hits && (!x || !y || !z))
        return hte::report(HT_E_INVAL, "hit arrays must not be NULL");
    if (n_hits > sec->max_hits)
        return hte::report(HT_E_INVAL, "more hits than max_hits");
    cudaStream_t st = stream ? (cudaStream_t)stream : sec->stream;
    return in_order(sec, st, [&] { return ht_fill(sec->ctx, x, y, z, n_hits, flags, st); });
}

ht_status ht_sectors_find_maxima(ht_sectors *sec, ht_peak *out, uint32_t capacity, uint32_t *n_found,
                                 uint32_t flags, void *stream)
{
    hte::TraceRange tr("ht_sectors_find_maxima");
    ht_status s = check_sec(sec);
    if (s != HT_OK)
        return s;
    if (flags & ~(uint32_t)HT_MEM_DEVICE)
        return hte::report(HT_E_INVAL, "unknown flag");
    if (!n_found || (capacity && !out))
        return hte::report(HT_E_INVAL, "out (capacity > 0) and n_found must not be NULL");
    cudaStream_t st = stream ? (cudaStream_t)stream : sec->stream;
    return in_order(sec, st, [&] { return ht_find_maxima(sec->ctx, out, capacity, n_found, flags, st); });
}

ht_status ht_sectors_copy_matrix(ht_sectors *sec, uint32_t sector, uint32_t *dst, uint64_t n_cells)
{
    ht_status s = check_sec(sec);
    if (s != HT_OK)
        return s;
    if (sector >= sec->S)
        return hte::report(HT_E_INVAL, "sector out of range");
    const hte::Engine &E = hte::ctx_engine(sec->ctx);
    const uint64_t slice = (uint64_t)E.geom.na * E.geom.nb, part = sec->m * slice;   // cells of a slice, of a theta row
    if (!dst || n_cells != E.geom.nt * part)
        return hte::report(HT_E_INVAL, "dst must hold exactly n_theta*n_phi*n_a*n_b cells");
    if (sec->done_pending)
        SCK(cudaStreamWaitEvent(sec->stream, sec->done, 0));   // the fill may have run on any stream
    for (uint32_t t = 0; t < E.geom.nt; ++t)
        SCK(cudaMemcpyAsync(dst + t * part, E.d_M + ((uint64_t)t * E.geom.np + (uint64_t)sector * sec->m) * slice,
                            part * 4, cudaMemcpyDeviceToHost, sec->stream));
    SCK(cudaStreamSynchronize(sec->stream));
    return HT_OK;
}

} // extern "C"
