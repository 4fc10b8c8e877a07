// flb_resident_batch.cu -- the resident kernel over the replicas of a batch.
#include "flb_resident_batch.cuh"

namespace flb {

namespace {

template <int SAMPLE>
struct ReplicaPar {
    using Store = float;
    using Key = KeyPairs;
    KeyPairs key;
    const CollidePairs& cc;
    const ReplicaHot& h;
    double s;
    // with FP32 products the deviation itself
    __device__ __forceinline__ f2 scaled(f2 f, int i) const {
        return SAMPLE == kResExact ? f - f2(h.ref[i]) : mad(f, f2(h.sinv), f2(h.snref[i]));
    }
    __device__ __forceinline__ float ref(int i) const { return h.ref[i]; }
    __device__ __forceinline__ f2 decode(f2 v, int) const { return v; }
    __device__ __forceinline__ f2 encode(f2 f, int) const { return f; }
};

template <int BASIS, int SAMPLE>
__global__ void __launch_bounds__(kResMaxWarps * 32, 1) resident_batch_kernel(const ResidentBatchArgs a) {
    extern __shared__ __align__(128) unsigned char res_smem[];
    ReplicaHot& h = *reinterpret_cast<ReplicaHot*>(res_smem);
    const ResCta e = a.table[blockIdx.x];
    const unsigned step = __ldcg(&a.ctl->step);
    {
        const uint32_t* from = reinterpret_cast<const uint32_t*>(&a.desc[e.slot].hot);
        for (int q = threadIdx.x; q < (int)(sizeof(ReplicaHot) / 4); q += blockDim.x)
            reinterpret_cast<uint32_t*>(res_smem)[q] = from[q];
    }
    __syncthreads();
    const int t = h.t0 + (int)(step - (unsigned)h.join);
    const int n = min(a.n, h.tend - t);   // a replica at its end stays there
    if (n > 0) {
        ResBlock k;
        k.src = h.buf[t & 1];
        k.dst = h.buf[(t + n) & 1];
        k.geo.Lx = h.Lx;
        k.geo.Ly = h.Ly;
        k.geo.pitch = h.pitch;
        k.geo.plane = h.plane;
        k.gx = 1;
        k.gy = e.gy;
        res_place(k, 0, e.iy);
        k.mail = a.mail + e.mail;
        k.mail_words = e.words;
        k.tag0 = a.tag0;
        k.t0 = (uint32_t)t;
        k.n = n;
        k.first = n;
        k.every = 1;
        if (SAMPLE != kResQuiet && h.every > 0) {
            const int since = t - h.warmup;
            k.first = since < 0 ? -since : (h.every - since % h.every) % h.every;
            k.every = h.every;
        }
        k.acc = h.acc;
        k.err = h.err;
        k.lut = a.lut;
        k.fields = nullptr;
        k.ffirst = k.fevery = n;
        resident_run<BASIS, SAMPLE>(k, ReplicaPar<SAMPLE>{KeyPairs(h.cc.key), h.pc, h, SAMPLE == kResExact ? 1.0 : (double)h.gram_s}, res_smem + kResHotBytes);
    }
    // the last CTA to finish advances the batch step (every CTA read it at its start)
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&a.ctl->ticket, 1u) == gridDim.x - 1) {
            a.ctl->step = step + (unsigned)a.n;
            a.ctl->ticket = 0u;
        }
    }
}

template <int BASIS>
const void* of_mode(int mode) {
    return mode == kResQuiet    ? (const void*)resident_batch_kernel<BASIS, kResQuiet>
           : mode == kResStaged ? (const void*)resident_batch_kernel<BASIS, kResStaged>
                                : (const void*)resident_batch_kernel<BASIS, kResExact>;
}

}  // namespace

const void* resident_batch_kernel_for(int basis, int mode) {
    return basis == 0 ? of_mode<0>(mode) : basis == 1 ? of_mode<1>(mode) : of_mode<2>(mode);
}

}  // namespace flb
