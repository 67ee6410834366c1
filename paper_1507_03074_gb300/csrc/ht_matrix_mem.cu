// Device memory of the vote matrices.
//
// M_H is written whole by every fill and is nearly empty (4.5 % of the cells
// of a paper-scale event hold a vote), and the fills are bound by that write.
// In memory asked for as compressible the L2 keeps and writes back such lines
// compressed: fewer bytes reach HBM, and every reader sees the same contents.
// The driver calls are looked up at run time, so the library loads where no
// driver is installed; wherever one of them is missing or refuses, the memory
// is ordinary cudaMalloc memory.
//
// Measured (bulk copies of 16 KB, back to back, one word in 22 nonzero): 256
// MiB written in 36.9 us against 43.2 us in ordinary memory and read in 18.7
// against 39.1 us, 4 GiB written in 515 against 645 us.  That holds for a grid
// that writes neighbouring tiles at any time, as the tile fill does; with a
// range per CTA, gigabytes apart, 4 GiB take 820 us against 645, which is why
// only the matrices of binnings that the tile fill serves are placed so.
#include "ht_engine.h"

#include <cuda.h>

namespace hte {

namespace {

struct DriverCalls {
    decltype(&cuDeviceGet) device_get = nullptr;
    decltype(&cuDeviceGetAttribute) attribute = nullptr;
    decltype(&cuMemGetAllocationGranularity) granularity = nullptr;
    decltype(&cuMemCreate) create = nullptr;
    decltype(&cuMemRelease) release = nullptr;
    decltype(&cuMemAddressReserve) reserve = nullptr;
    decltype(&cuMemAddressFree) unreserve = nullptr;
    decltype(&cuMemMap) map = nullptr;
    decltype(&cuMemUnmap) unmap = nullptr;
    decltype(&cuMemSetAccess) set_access = nullptr;
    bool ok = false;

    template <class F>
    static bool look_up(const char *name, F *f)
    {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess || !p) {
            cudaGetLastError();
            return false;
        }
        *f = reinterpret_cast<F>(p);
        return true;
    }
    DriverCalls()
    {
        ok = look_up("cuDeviceGet", &device_get) && look_up("cuDeviceGetAttribute", &attribute) &&
             look_up("cuMemGetAllocationGranularity", &granularity) && look_up("cuMemCreate", &create) &&
             look_up("cuMemRelease", &release) && look_up("cuMemAddressReserve", &reserve) &&
             look_up("cuMemAddressFree", &unreserve) && look_up("cuMemMap", &map) &&
             look_up("cuMemUnmap", &unmap) && look_up("cuMemSetAccess", &set_access);
    }
};

const DriverCalls &driver()
{
    static const DriverCalls d;
    return d;
}

// Compressible memory mapped for `device` alone (as cudaMalloc's is), or false.
bool map_compressible(MatrixMem &m, size_t bytes, int device)
{
    const DriverCalls &d = driver();
    CUdevice dev;
    int supported = 0;
    if (!d.ok || d.device_get(&dev, device) != CUDA_SUCCESS ||
        d.attribute(&supported, CU_DEVICE_ATTRIBUTE_GENERIC_COMPRESSION_SUPPORTED, dev) != CUDA_SUCCESS || !supported)
        return false;
    CUmemAllocationProp prop{};
    prop.type = CU_MEM_ALLOCATION_TYPE_PINNED;
    prop.location.type = CU_MEM_LOCATION_TYPE_DEVICE;
    prop.location.id = device;
    prop.allocFlags.compressionType = CU_MEM_ALLOCATION_COMP_GENERIC;
    size_t gran = 0;
    if (d.granularity(&gran, &prop, CU_MEM_ALLOC_GRANULARITY_RECOMMENDED) != CUDA_SUCCESS || !gran)
        return false;
    const size_t size = (bytes + gran - 1) / gran * gran;
    CUmemGenericAllocationHandle h;
    if (d.create(&h, size, &prop, 0) != CUDA_SUCCESS)
        return false;
    CUdeviceptr va = 0;
    bool ok = d.reserve(&va, size, 0, 0, 0) == CUDA_SUCCESS;
    if (ok && d.map(va, size, 0, h, 0) != CUDA_SUCCESS) {
        d.unreserve(va, size);
        ok = false;
    }
    d.release(h);   // a mapping keeps the memory
    if (!ok)
        return false;
    CUmemAccessDesc acc{};
    acc.location = prop.location;
    acc.flags = CU_MEM_ACCESS_FLAGS_PROT_READWRITE;
    if (d.set_access(va, size, &acc, 1) != CUDA_SUCCESS) {
        d.unmap(va, size);
        d.unreserve(va, size);
        return false;
    }
    m.p = reinterpret_cast<uint32_t *>(va);
    m.mapped = size;
    return true;
}

} // namespace

cudaError_t matrix_alloc(MatrixMem &m, size_t bytes, int device, bool compressible)
{
    m = MatrixMem{};
    if (compressible && bytes >= kCompressMin && map_compressible(m, bytes, device))
        return cudaSuccess;
    return cudaMalloc(reinterpret_cast<void **>(&m.p), bytes);
}

void matrix_free(MatrixMem &m, void *guard)
{
    const cudaError_t waited = cudaFree(guard);
    if (m.mapped) {
        // Freeing the guard waits for every kernel and copy of the device that owns
        // it, whichever device is current, and may run beside another thread's
        // stream capture, which a device synchronisation would break.  Where it
        // fails the memory stays mapped: something may still use it.  (The guard is
        // a block that the engine has anyway: one of the matrix's own, allocated in
        // front of it, moved the small buffers and cost the upgrade event 1.2 %.)
        const DriverCalls &d = driver();
        const CUdeviceptr va = reinterpret_cast<CUdeviceptr>(m.p);
        if (waited == cudaSuccess && d.unmap(va, m.mapped) == CUDA_SUCCESS)
            d.unreserve(va, m.mapped);
    } else {
        cudaFree(m.p);
    }
    m = MatrixMem{};
}

} // namespace hte
