// How many pages an event has. Plain C++, so that it can also be compiled for the host by itself.
#pragma once

#ifdef __CUDACC__
#define AKV_PAGES_HD __host__ __device__ __forceinline__
#else
#define AKV_PAGES_HD inline
#endif

namespace akv {

// N slots (at least one) in pages of 2^shift of them, up to 2^30. Page numbers are compared with this, never first slots: one page can hold more
// slots than the event has, and (page << shift) of a page that the event does not have need not fit an int.
AKV_PAGES_HD int event_pages(int N, int shift) { return ((N - 1) >> shift) + 1; }

}  // namespace akv
