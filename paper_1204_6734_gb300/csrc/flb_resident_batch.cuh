// flb_resident_batch.cuh -- the resident kernel (flb_resident.cuh) over the
// replicas of a batch: CTA b steps block `iy` of `gy` rows of blocks of replica
// `slot` of its table entry, n steps in one launch.
//
// Small replicas take one CTA each, with as many CTAs on an SM as their number
// asks for (up to four of four warps): they need no one, so there may be more
// of them than fit at once. Where there are fewer replicas than SMs the larger
// ones are cut into rows of blocks that exchange through mailboxes, all CTAs
// resident at once (cooperative launch).
#pragma once

#include "flb_batch_kernel.cuh"
#include "flb_resident.cuh"

namespace flb {

struct ResCta {
    uint32_t slot;
    int gy, iy;
    int mail;        // first mailbox word of the replica
    int words;       // words of one of its two mailboxes
};

struct ResidentBatchArgs {
    const ReplicaDesc* desc;
    const ResCta* table;
    BatchCtl* ctl;
    const float* lut;
    uint64_t* mail;
    uint32_t tag0;
    int n;
};

// Sampling mode and basis of the kernel (flb_resident_batch.cu).
const void* resident_batch_kernel_for(int basis, int mode);

constexpr size_t kResHotBytes = (sizeof(ReplicaHot) + 15) / 16 * 16;

}  // namespace flb
