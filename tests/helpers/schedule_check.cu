// Test helper: the library's count of sampled steps (flb_host.h), on the host.
#include "../../paper_1204_6734_gb300/csrc/flb_host.h"

extern "C" long long sampled(long long ta, long long tb, long long warmup, long long every) {
    return flb::count_sampled(ta, tb, warmup, every);
}
