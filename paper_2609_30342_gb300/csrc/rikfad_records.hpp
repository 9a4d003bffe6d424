// rikfad_records.hpp -- which recorded step of a quadratic run comes next.
// Plain integer logic shared by the kernels and by a host check of the loop
// that it drives (its end must not depend on the list, which is device memory
// that the host never sees).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define RK_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define RK_HOST_DEVICE inline
#endif

namespace rikfad {

// First index r with record[r] >= k (record ascending).
RK_HOST_DEVICE int64_t first_record_at_or_after(const int64_t *record, int64_t nrecord, int64_t k)
{
    int64_t lo = 0, hi = nrecord;
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (record[mid] < k)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Step of record[r] relative to the launch start k0, or -1 when there is none
// from step s to the launch's last.  An entry behind s (a list out of order) is
// none: the kernels run up to the step returned here, so one that they have
// passed would never come.
RK_HOST_DEVICE int record_in_launch(const int64_t *record, int64_t nrecord, int64_t r, int64_t k0, int s, int steps)
{
    if (r >= nrecord)
        return -1;
    const int64_t rel = record[r] - k0;
    return (uint64_t)(rel - s) <= (uint64_t)(steps - s) ? (int)rel : -1;    // s <= rel <= steps
}

}  // namespace rikfad
