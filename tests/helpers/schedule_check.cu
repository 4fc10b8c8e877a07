// Test helper: the library's count of sampled steps (flb_host.h), on the host.
#include "../../paper_1204_6734_gb300/csrc/flb_host.h"

extern "C" long long sampled(long long ta, long long tb, long long warmup, long long every) {
    return flb::count_sampled(ta, tb, warmup, every);
}

// Whether an error at (step, node) of a launch of n steps from t0 replaces a recorded one.
extern "C" int precedes(int code, long long had_node, long long had_step, long long node, unsigned step, unsigned t0, int n) {
    flb::DevError had{};
    had.code = code;
    had.node = had_node;
    had.step = had_step;
    return flb::error_precedes(had, node, step, t0, n);
}

// alloc_with_extra over a device with `free` bytes: the bytes it got (-1: an error), and
// whether the extra ones are among them.
extern "C" long long extra(long long free, long long need, long long extra_bytes, int* got) {
    void* p;
    bool with = false;
    long long bytes = -1;
    const auto alloc = [&](void** q, size_t n) {
        if ((long long)n > free) return cudaErrorMemoryAllocation;
        bytes = (long long)n;
        *q = &bytes;
        return cudaSuccess;
    };
    const cudaError_t ce = flb::alloc_with_extra(alloc, &p, (size_t)need, (size_t)extra_bytes, &with);
    *got = with;
    return ce == cudaSuccess && p ? bytes : -1;
}
