// Host memory that copies from the device are about to fill.
#pragma once
#include <cstddef>
#include <cstdint>
#include <sys/mman.h>
#include <unistd.h>

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23  // Linux 5.14
#endif

namespace tlb {

// Maps the pages of a pageable buffer without touching what they hold: the
// buffer belongs to the caller until the stream reaches the copies (an upload
// from it may still be queued), so nothing is stored to it.  Without its pages
// the device takes the faults of a fresh buffer one by one: GB300, 6 FP64 planes
// of 192x96x192 (170 MB) into a new numpy array 75 -> 6.0 ms, of 64^3 2.5 -> 0.55
// ms, 5 planes of 2048x2048 6.4 -> 6.0 ms.  A buffer whose pages are there
// already is told by a few of them (the whole walk takes 0.5 ms of the 1.2 that
// such a read-out of 170 MB takes).  Where the kernel does not know the call, or
// refuses it, the copies take the faults.
inline int map_host_pages(void* p, size_t bytes)
{
    if (!bytes) return 0;
    const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    const uintptr_t a = (uintptr_t)p / page, n = ((uintptr_t)p + bytes + page - 1) / page - a;
    const uintptr_t looks = n < 4 ? n : 4;
    for (uintptr_t i = 0; i < looks; i++) {
        const uintptr_t at = a + (looks == 1 ? 0 : i * (n - 1) / (looks - 1));
        unsigned char there = 0;
        if (mincore((void*)(at * page), page, &there) != 0 || !(there & 1))
            return madvise((void*)(a * page), n * page, MADV_POPULATE_WRITE);
    }
    return 0;
}

}  // namespace tlb
