// sssp_small.cu -- the single-query small-round kernels of sssp_small.cuh for
// the two state layouts, label-setting and windowed.
#include "sssp_engine.h"
#include "sssp_small.cuh"

namespace sssp {

TailKernel small_kernel(bool narrow, bool win) {
    TailKernel k;
    if (narrow)
        k.fn = win ? (const void*)k_small<SmallNarrow, true> : (const void*)k_small<SmallNarrow, false>;
    else
        k.fn = win ? (const void*)k_small<SmallWide, true> : (const void*)k_small<SmallWide, false>;
    k.threads = kSmallThreads;
    k.smem = sizeof(SmallShared);
    return k;
}

}  // namespace sssp
