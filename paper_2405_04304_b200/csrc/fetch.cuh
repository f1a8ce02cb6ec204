// The inputs of an iteration from pinned host memory to the context's buffers, by one small kernel.
//
// Bound: the latency of one round trip over PCIe, then its bandwidth; every thread has its one load in flight at once.  A copy
// by the copy engine in the stream keeps the kernel behind it from being launched early; this one lets the draft phase set
// itself up and request the LM head while the hidden states arrive.  It looks at the caller's memory only once the work before
// it in the stream is done, as a copy there would: that work may be what writes the hidden states.
#pragma once

#include "common.cuh"

namespace disco {

constexpr int kFetchThreads = 64;   // (few registers and no shared memory: fits beside the kernel that follows)
struct FetchPart {
    const void* src;    // host memory as the device sees it
    void* dst;
    unsigned pieces;    // of 16 bytes, or of 4
    unsigned wide;
};
struct FetchParams {
    FetchPart part[5];
    int n;
};

static __global__ void __launch_bounds__(kFetchThreads) fetch_kernel(const FetchParams p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");   // (every thread: no part of this kernel ends before what went before it)
    unsigned i = blockIdx.x * kFetchThreads + threadIdx.x;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (k >= p.n) break;
        const unsigned pieces = p.part[k].pieces;
        if (i < pieces) {
            if (p.part[k].wide) __stcg(static_cast<uint4*>(p.part[k].dst) + i, __ldcv(static_cast<const uint4*>(p.part[k].src) + i));
            else __stcg(static_cast<uint32_t*>(p.part[k].dst) + i, __ldcv(static_cast<const uint32_t*>(p.part[k].src) + i));
            break;
        }
        i -= pieces;
    }
}

}  // namespace disco
