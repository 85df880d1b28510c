// Copies of results into the caller's memory.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include <sys/mman.h>
#include <unistd.h>

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23  // Linux 5.14
#endif

namespace pa {

// Brings the pages of [p, p + bytes) into memory, writable, without writing to them.  Pages that the
// caller may not write, or that are not there, stay as they are: they are the copy's to meet.
inline void populate_pages(void *p, size_t bytes)
{
    const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    const uintptr_t lo = (uintptr_t)p & ~(page - 1), hi = ((uintptr_t)p + bytes + page - 1) & ~(page - 1);
    (void)madvise(reinterpret_cast<void *>(lo), hi - lo, MADV_POPULATE_WRITE);
}

// Enqueues the copy of a result into the caller's memory, whose pages are first populated from the
// host, while the device still works on the result.  A copy into pages that have never been touched
// takes their faults one by one from the device: 20.8 MB into fresh pages 17 ms, 0.8 ms after
// populating them (0.13 ms into pages in use).  Only pageable memory is populated: pinned pages are
// there already.
inline cudaError_t copy_out(void *host, const void *dev, size_t bytes, cudaStream_t s)
{
    if (bytes >= (1u << 20)) {
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, host) != cudaSuccess)
            (void)cudaGetLastError();  // of this query alone: the copy says what is wrong with the pointer
        else if (at.type == cudaMemoryTypeUnregistered)
            populate_pages(host, bytes);
    }
    return cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, s);
}

}  // namespace pa
