// Host-side helpers of the library that need neither a kernel nor a device.
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <cstddef>
#include <cstdint>

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23
#endif

namespace pff {

// Map the pages of a host buffer that the device is about to write, without changing what they hold (the copy
// may still fail). The device copies straight into pageable memory here, and pages that are not mapped yet (a fresh
// numpy array) are faulted in from its side: Rve.get of 100 MB 4.5 -> 3.5 ms, of 0.1 MB 0.13 -> 0.05 ms, and
// nothing on pages that are mapped (0.63 ms for 100 MB; a store to every 4 KB cost 0.18 ms there). One call for the
// range, whatever the page size. A hint: where it is refused (an older kernel, memory that is not ordinary host
// memory) the copy does without.
inline void map_pages(void *p, size_t bytes) {
    static const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    if (!p || !bytes) return;
    const uintptr_t a = (uintptr_t)p & ~(page - 1), e = ((uintptr_t)p + bytes + page - 1) & ~(page - 1);
    (void)madvise((void *)a, e - a, MADV_POPULATE_WRITE);
}

}  // namespace pff
