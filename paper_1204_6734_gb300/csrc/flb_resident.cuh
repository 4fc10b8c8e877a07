// flb_resident.cuh -- many time steps per launch of an FP32 lattice whose
// populations stay in shared memory between the steps.
//
// The lattice is cut into gx x gy blocks, one CTA each (one block: the whole
// lattice in one CTA). A CTA loads the pre-collision populations of its nodes
// once, steps them n times and stores the result once, in the ghost-frame
// layout of every other kernel. Against one launch per step this saves the
// launch, the pipeline's start and its end in every step (7 to 9 us of the
// 8.1 us that a step of a 21 x 21 lattice took, of 10 us at 300 x 130 and of
// 20 us at 1000 x 750) and the trip of 72 bytes per node through L2 or HBM.
//
// In place: one copy of the populations, cell (X, Y, i) at (X + bw Y) 9 + i
// (stride 9 words: no bank conflicts). s steps after the load, f_i of node
// (x, y) sits in cell ((x - s v_ix) mod bw, (y - s v_iy) mod bh): the node
// reads its nine cells, collides and writes f*_i back to the same nine cells,
// and because the offsets have moved on by one, the next step's read of node
// x + v_i is that cell. Streaming costs no copy, no cell is touched by two
// threads in a step, one barrier per step orders the steps, and the wrap of
// the offsets is the periodic boundary where the lattice is not cut.
//
// Cells are addressed in bytes of shared memory: a pair's three column and three
// row offsets (each the smaller of two unsigned sums) give its 18 addresses by
// one addition or subtraction each, and what rarely is asked for (a node's place
// in the lattice) is divided out where it is. As word indices into an array
// the same took 16.1 instructions per node against 12.4 in the one-step kernel;
// us per step with those and with these: 21 x 21 2.18 / 2.08, 300 x 130 4.27 / 4.13, 1000 x
// 750 16.4 / 15.7, 384 x 21^2 6.25 / 5.90 (with all that this file does by now 2.06, 4.11,
// 15.1, 5.30).
//
// Node pairs (packed FP32x2): node A is the m-th of the block, node B the m-th
// from its end, i.e. (bw - 1 - x, bh - 1 - y), so B's cells follow from A's
// by one subtraction each (cell_i(B) = nn - 1 - cell_opposite(i)(A)), and the
// block's first and last row are done first, in the same pass: what they send
// is under way while the rows between them are computed.
//
// Between blocks: a population that leaves its block is written, besides, to a
// mailbox in global memory as one 64-bit word {value, tag}, tag = a number
// that grows with every step and launch of the handle. The reader polls the
// word itself until the tag is the one of its step: one trip through L2, no
// fence and no flag. Two mailboxes alternate; a word of one is overwritten
// two steps later, by a node that has by then received the populations of the
// very nodes that read it, so no reader can be overtaken. All CTAs are
// resident at once (cooperative launch), every wait is bounded (flb_tma.cuh).
//
// Correlation sums: as flb_gram.cuh (staged in FP16 for the tensor cores, or with
// FP32 products where a batch's tile shape promises them and for the FP16 store),
// except that every step's FP32 partials (at most 1024 products per warp) go to FP64
// by themselves, in a fixed order: the sums do not depend on how many steps a launch
// makes.
#pragma once

#include <cuda_runtime.h>

#include "flb_collide.cuh"
#include "flb_gram.cuh"
#include "flb_kernels.cuh"
#include "flb_pipeline.cuh"
#include "flb_layout.cuh"
#include "flb_tma.cuh"

namespace flb {

constexpr int kResMaxWarps = 16;   // 512 threads of 128 registers
constexpr int kResSlot = 96;       // floats per warp and parity

// Sampling of a resident launch: none; deviations staged in FP16; FP32 products.
enum : int { kResQuiet = 0, kResStaged = 1, kResExact = 2 };
// Entries kept: of the Gram matrix rows 0..7 x columns 0..9 and rows 8, 9 x 8, 9.
__host__ __device__ constexpr int res_entries(int mode) { return mode == kResExact ? kProdEntries : 84; }

__host__ __device__ constexpr size_t res_cells_bytes(int cells) { return ((size_t)cells * 36 + 15) / 16 * 16; }
__host__ __device__ constexpr size_t res_sample_bytes(int mode, int warps) {
    return mode == kResQuiet ? 0
                             : (size_t)warps * ((mode == kResExact ? kProdWarpFloats * 4 : kGramWarpHalves * 2) + 2 * kResSlot * 4) +
                                   kResSlot * 8;
}
// Dynamic shared memory of a CTA of `warps` warps holding `cells` nodes.
__host__ __device__ constexpr size_t res_smem_bytes(int cells, int mode, int warps) {
    return res_cells_bytes(cells) + res_sample_bytes(mode, warps) + 16;
}

// One CTA's block of one lattice and what to do with it.
struct ResBlock {
    const void* src;        // holds f*(t0 - 1), in the store's type
    void* dst;              // receives f*(t0 + n - 1)
    Geometry geo;
    int x0, y0, bw, bh;
    int gx, gy, ix, iy;     // the block's place in the grid of blocks
    uint64_t* mail;         // two mailboxes of mail_words words (gx gy > 1)
    int mail_words;
    uint32_t tag0;          // tag of the state at t0
    uint32_t t0;
    int n;
    int first, every;       // steps of this launch sampled: first, first + every, ...
    double* acc;
    DevError* err;
    const float* lut;
    float* fields;          // structure-factor fields (3 Lx Ly values each) of the states at
    int ffirst, fevery;     // t0 + ffirst, t0 + ffirst + fevery, ... (or null)
};

__device__ __forceinline__ uint64_t ld_mail(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_mail(uint64_t* p, float v, uint32_t tag) {
    const uint64_t w = (uint64_t)tag << 32 | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

// Place of population i among the three that cross a y (x) boundary together.
__host__ __device__ constexpr int res_ky(int i) { return i == 2 || i == 4 ? 0 : (i == 5 || i == 7 ? 1 : 2); }
__host__ __device__ constexpr int res_kx(int i) { return i == 1 || i == 3 ? 0 : (i == 5 || i == 6 ? 1 : 2); }
__host__ __device__ constexpr int opposite(int i) { return i == 0 ? 0 : (i < 5 ? (i + 1) % 4 + 1 : (i - 3) % 4 + 5); }
static_assert(opposite(1) == 3 && opposite(2) == 4 && opposite(3) == 1 && opposite(4) == 2 && opposite(5) == 7 &&
                  opposite(6) == 8 && opposite(7) == 5 && opposite(8) == 6,
              "opposite velocities");

// Words of one mailbox: the y boundaries (upwards, downwards), Lx columns of
// three populations each, then the x boundaries, Ly rows.
inline long long res_mail_words(int Lx, int Ly, int gx, int gy) {
    return (gy > 1 ? 6LL * gy * Lx : 0) + (gx > 1 ? 6LL * gx * Ly : 0);
}

// Which edges of its block node A of a pair lies on (only edges where the
// lattice is cut). Node B, the pair's image, lies on the opposite ones and
// exchanges the opposite populations there.
struct ResEdge {
    bool l, r, b, t;
    __device__ __forceinline__ bool any() const { return l || r || b || t; }
};

// The boundaries of one axis between the blocks: g of them, the CTA's block j,
// lines of n nodes; the words start at `first`.
struct ResAxis {
    int g, j, n, first;
};

// Mailbox word of population I pulled by (In) or leaving from (!In) a node at u
// along a boundary of axis AXIS (1: y boundaries, u the node's X; 0: x, its Y).
// The word belongs to the sender: the direction, the sender's block, the
// population, the sender's u.
template <int AXIS, int I, bool In>
__device__ __forceinline__ int res_word(const ResAxis& b, int u) {
    constexpr int across = AXIS ? cvy(I) : cvx(I), along = AXIS ? cvx(I) : cvy(I), k = AXIS ? res_ky(I) : res_kx(I);
    const int j = In ? wrap(b.j - across, b.g) : b.j;
    return b.first + (((across > 0 ? 0 : b.g) + j) * 3 + k) * b.n + (In ? wrap(u - along, b.n) : u);
}

template <class T>
__device__ __forceinline__ void store_lane(T* p, const Geometry& geo, int x, int y, const f2 f[9], int k) {
    T v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = (T)lane(f[i], k);
    store_node_ghosts(p, geo, x, y, v);
}

// Shared-memory cells by 32-bit address; population I of a cell is 4 I bytes in.
template <int I>
__device__ __forceinline__ float cell_load(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(4 * I) : "memory");
    return v;
}
template <int I>
__device__ __forceinline__ void cell_store(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(a), "n"(4 * I), "f"(v) : "memory");
}

// The nine cells of node A from its column and row offsets (bytes; the columns
// hold the address of cell 0), and node B's from them.
struct ResCells {
    uint32_t r[3], c[3];   // index v + 1
    uint32_t kb;           // twice the address of cell 0, plus 36 (nn - 1)
    template <int I>
    __device__ __forceinline__ uint32_t a() const { return r[cvy(I) + 1] + c[cvx(I) + 1]; }
    template <int I>
    __device__ __forceinline__ uint32_t b() const { return kb - (r[1 - cvy(I)] + c[1 - cvx(I)]); }
    template <int I>
    __device__ __forceinline__ f2 load() const { return f2(cell_load<I>(a<I>()), cell_load<I>(b<I>())); }
};

__device__ __forceinline__ void load_cells(const ResCells& a, f2 (&g)[9]) {
    g[0] = a.load<0>();
    g[1] = a.load<1>();
    g[2] = a.load<2>();
    g[3] = a.load<3>();
    g[4] = a.load<4>();
    g[5] = a.load<5>();
    g[6] = a.load<6>();
    g[7] = a.load<7>();
    g[8] = a.load<8>();
}

template <int I>
__device__ __forceinline__ void store_cell(const ResCells& a, const f2 (&f)[9], bool both) {
    cell_store<I>(a.a<I>(), f[I].v.x);
    if (both) cell_store<I>(a.b<I>(), f[I].v.y);
}
__device__ __forceinline__ void store_cells(const ResCells& a, const f2 (&f)[9], bool both) {
    store_cell<0>(a, f, both);
    store_cell<1>(a, f, both);
    store_cell<2>(a, f, both);
    store_cell<3>(a, f, both);
    store_cell<4>(a, f, both);
    store_cell<5>(a, f, both);
    store_cell<6>(a, f, both);
    store_cell<7>(a, f, both);
    store_cell<8>(a, f, both);
}

// Receive across one edge: A's populations I0, I1, I2 (cells a0..a2, A at u
// along the edge) and B's opposite ones (b0..b2, v), once all carry the step's
// tag. skip1, skip2: I1, I2 cross the other axis' boundary, too, and came from
// there. Not inlined, and all arguments scalars: references put the block and the
// cells into local memory for the whole step (176 bytes a thread; us per step with
// them and without: 300 x 130 4.11 / 4.02, 1000 x 750 15.66 / 15.16).
template <int AXIS, int I0, int I1, int I2>
__device__ __noinline__ void res_receive(const uint64_t* in, uint32_t tag, int g, int j, int n, int first, int u, int v,
                                         uint32_t a0, uint32_t a1, uint32_t a2, uint32_t b0, uint32_t b1, uint32_t b2,
                                         bool skip1, bool skip2, volatile int* gave_up) {
    const ResAxis ax{g, j, n, first};
    const uint64_t* pa0 = in + res_word<AXIS, I0, true>(ax, u);
    const uint64_t* pa1 = in + res_word<AXIS, I1, true>(ax, u);
    const uint64_t* pa2 = in + res_word<AXIS, I2, true>(ax, u);
    const uint64_t* pb0 = in + res_word<AXIS, opposite(I0), true>(ax, v);
    const uint64_t* pb1 = in + res_word<AXIS, opposite(I1), true>(ax, v);
    const uint64_t* pb2 = in + res_word<AXIS, opposite(I2), true>(ax, v);
    const uint64_t have = (uint64_t)tag << 32;
    uint64_t wa0, wa1 = have, wa2 = have, wb0, wb1 = have, wb2 = have;
    long long began = 0;
    while (true) {
        wa0 = ld_mail(pa0);
        wb0 = ld_mail(pb0);
        if (!skip1) {
            wa1 = ld_mail(pa1);
            wb1 = ld_mail(pb1);
        }
        if (!skip2) {
            wa2 = ld_mail(pa2);
            wb2 = ld_mail(pb2);
        }
        const uint32_t bad = ((uint32_t)(wa0 >> 32) ^ tag) | ((uint32_t)(wb0 >> 32) ^ tag) |
                             ((uint32_t)(wa1 >> 32) ^ tag) | ((uint32_t)(wb1 >> 32) ^ tag) |
                             ((uint32_t)(wa2 >> 32) ^ tag) | ((uint32_t)(wb2 >> 32) ^ tag);
        if (bad == 0 || *gave_up) break;
        if (began == 0) {
            began = clock64();
        } else if (clock64() - began > kWaitCycles) {
            gave_up[1] = (int)tag;
            *gave_up = 1;
            break;
        }
    }
    cell_store<I0>(a0, __uint_as_float((uint32_t)wa0));
    cell_store<opposite(I0)>(b0, __uint_as_float((uint32_t)wb0));
    if (!skip1) {
        cell_store<I1>(a1, __uint_as_float((uint32_t)wa1));
        cell_store<opposite(I1)>(b1, __uint_as_float((uint32_t)wb1));
    }
    if (!skip2) {
        cell_store<I2>(a2, __uint_as_float((uint32_t)wa2));
        cell_store<opposite(I2)>(b2, __uint_as_float((uint32_t)wb2));
    }
}

// Send across one edge: A's populations I0, I1, I2 and (unless B is A) B's
// opposite ones, read back from the pair's cells.
template <int AXIS, int I0, int I1, int I2>
__device__ __noinline__ void res_send(uint64_t* out, uint32_t tag, int g, int j, int n, int first, int u, int v,
                                      uint32_t a0, uint32_t a1, uint32_t a2, uint32_t b0, uint32_t b1, uint32_t b2,
                                      bool skip1, bool skip2, bool both) {
    const ResAxis ax{g, j, n, first};
    st_mail(out + res_word<AXIS, I0, false>(ax, u), cell_load<I0>(a0), tag);
    if (!skip1) st_mail(out + res_word<AXIS, I1, false>(ax, u), cell_load<I1>(a1), tag);
    if (!skip2) st_mail(out + res_word<AXIS, I2, false>(ax, u), cell_load<I2>(a2), tag);
    if (!both) return;
    st_mail(out + res_word<AXIS, opposite(I0), false>(ax, v), cell_load<opposite(I0)>(b0), tag);
    if (!skip1) st_mail(out + res_word<AXIS, opposite(I1), false>(ax, v), cell_load<opposite(I1)>(b1), tag);
    if (!skip2) st_mail(out + res_word<AXIS, opposite(I2), false>(ax, v), cell_load<opposite(I2)>(b2), tag);
}

// The calls for one edge of a pair.
template <int AXIS, int I0, int I1, int I2>
__device__ __forceinline__ void res_edge_in(const uint64_t* in, uint32_t tag, const ResAxis& ax, int u, int v,
                                            const ResCells& a, bool skip1, bool skip2, volatile int* gave_up) {
    res_receive<AXIS, I0, I1, I2>(in, tag, ax.g, ax.j, ax.n, ax.first, u, v, a.a<I0>(), a.a<I1>(), a.a<I2>(),
                                  a.b<opposite(I0)>(), a.b<opposite(I1)>(), a.b<opposite(I2)>(), skip1, skip2, gave_up);
}
template <int AXIS, int I0, int I1, int I2>
__device__ __forceinline__ void res_edge_out(uint64_t* out, uint32_t tag, const ResAxis& ax, int u, int v,
                                             const ResCells& a, bool skip1, bool skip2, bool both) {
    res_send<AXIS, I0, I1, I2>(out, tag, ax.g, ax.j, ax.n, ax.first, u, v, a.a<I0>(), a.a<I1>(), a.a<I2>(),
                               a.b<opposite(I0)>(), a.b<opposite(I1)>(), a.b<opposite(I2)>(), skip1, skip2, both);
}

// A warp's FP32 partials of one step: with FP32 products in prod_entry's order, else
// in the order of the kept entries (C is symmetric): rows 0..7 by columns 0..7, rows 0..7 by columns 8 and 9, rows 8
// and 9 by columns 8 and 9. Cleared for the next sampled step.
template <int SAMPLE>
__device__ __forceinline__ void res_publish(float (&c)[8], float* slot) {
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    if constexpr (SAMPLE == kResExact) {
        const float4 v = prod_take(c);
        if (lane < kProdBlocks) *reinterpret_cast<float4*>(slot + 4 * lane) = v;
        return;
    }
    *reinterpret_cast<float2*>(slot + 2 * lane) = make_float2(c[0], c[1]);
    if (q == 0) {
        *reinterpret_cast<float2*>(slot + 64 + 2 * g) = make_float2(c[4], c[5]);
        if (g < 2) *reinterpret_cast<float2*>(slot + 80 + 2 * g) = make_float2(c[6], c[7]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = 0.f;
}

// The CTA's sum of a step's partials of nw warps, added to the FP64 entries by
// the last 96 threads of the CTA (warps without nodes of their own where the
// block leaves room for them; entry q always by the same thread). All loads are
// under way before the first add: this sits in the step's critical path. The
// partials are added as FP64 would add them (to 2^-46): every FP32 addition's
// rounding error is kept and added up beside the sum; sixteen conversions and
// additions in FP64 would take 0.7 us of the pipe that this GPU has for them.
template <int SAMPLE>
__device__ __forceinline__ void res_reduce(const float* slots, double* red, int nw) {
    const int T = blockDim.x, r0 = T > kResSlot ? T - kResSlot : 0;
    for (int q = (int)threadIdx.x - r0; q >= 0 && q < res_entries(SAMPLE); q += T) {
        float v[kResMaxWarps], lo = 0.f;
#pragma unroll
        for (int w = 0; w < kResMaxWarps / 2; ++w) v[w] = w < nw ? slots[w * kResSlot + q] : 0.f;
        if (nw > kResMaxWarps / 2) {
#pragma unroll
            for (int w = kResMaxWarps / 2; w < kResMaxWarps; ++w) v[w] = w < nw ? slots[w * kResSlot + q] : 0.f;
#pragma unroll
            for (int w = 0; w < kResMaxWarps / 2; ++w) v[w] = two_sum(v[w], v[w + kResMaxWarps / 2], lo);
        }
#pragma unroll
        for (int h = kResMaxWarps / 4; h > 0; h >>= 1)
#pragma unroll
            for (int w = 0; w < h; ++w) v[w] = two_sum(v[w], v[w + h], lo);
        red[q] += (double)v[0] + (double)lo;
    }
}

// Sum q of the kSums layout from the kept entries.
template <int SAMPLE>
__device__ __forceinline__ double res_sum(const double* red, int q, double s) {
    if constexpr (SAMPLE == kResExact) return prod_sum(red, q, s);
    if (q < 9) return s * red[q < 8 ? 64 + 2 * q + 1 : 81];
    int k = q - 9, i = 0;
    while (k >= 9 - i) {
        k -= 9 - i;
        ++i;
    }
    const int j = i + k;
    return s * s * red[j < 8 ? 8 * i + j : (i < 8 ? 64 + 2 * i : 80)];
}

// Steps 0..n-1 of one block. Par: the lattice's parameters -- Store (the type in
// HBM; the cells hold the stored value as a float), decode(v, i) and encode(f,
// i) (from and to the stored value; encode rounds to the store), key, cc (the
// collision constants), s (the Gram scale), scaled(v, i) (the stored value's
// deviation in units of s), ref(i) (f_i^0(rho0, u0)).
template <int BASIS, int SAMPLE, bool CUT, class Par>
__device__ __forceinline__ void resident_run_of(const ResBlock& k, const Par& par, unsigned char* smem) {
    float* cell = reinterpret_cast<float*>(smem);
    const int T = blockDim.x, c = threadIdx.x, lane_id = c & 31, warp = c >> 5, nw = T >> 5;
    const int bw = k.bw, bh = k.bh, nn = bw * bh, pairs = (nn + 1) >> 1;
    const int nwork = min(nw, (pairs + 31) >> 5);   // warps with nodes
    const int Lx = k.geo.Lx;
    unsigned char* after = smem + res_cells_bytes(nn);
    double* red = reinterpret_cast<double*>(after);
    float* slots = reinterpret_cast<float*>(after + (SAMPLE ? kResSlot * 8 : 0));
    __half* gram = reinterpret_cast<__half*>(slots + (SAMPLE ? 2 * nw * kResSlot : 0));
    // {a wait gave up, its tag}, then the block's first error: step of the launch, node,
    // code (kStatusNonfinite: 1)
    volatile int* gave_up = reinterpret_cast<volatile int*>(after + res_sample_bytes(SAMPLE, nw));
    const auto first_error = [&] { return reinterpret_cast<unsigned long long*>(const_cast<int*>(gave_up) + 2); };
    if (c == 0) {
        *gave_up = 0;
        *first_error() = ~0ull;
    }

    constexpr bool kExact = SAMPLE == kResExact;
    const uint32_t blk = SAMPLE ? smem_u32(gram) + warp * (kExact ? kProdWarpFloats * 4 : kGramWarpHalves * 2) : 0u;
    const GramLane gh(kExact ? 0u : blk, kGramRows);
    const ProdLane gp(kExact ? blk : 0u);
    float gc[SAMPLE ? 8 : 1];
    if constexpr (SAMPLE != kResQuiet) {
#pragma unroll
        for (int q = 0; q < 8; ++q) gc[q] = 0.f;
        if constexpr (kExact)
            prod_init(reinterpret_cast<float*>(gram) + warp * kProdWarpFloats);
        else
            gram_init(gram + warp * kGramWarpHalves);
        for (int q = c - (T > kResSlot ? T - kResSlot : 0); q >= 0 && q < res_entries(SAMPLE); q += T) red[q] = 0.0;
    }

    // this thread's nodes: pairs c, c + T, ...
    const int dy = T / bw, dx = T - dy * bw;
    const int ys = c / bw, xs = c - ys * bw;
    const bool cutx = CUT && k.gx > 1, cuty = CUT && k.gy > 1;
    const ResAxis ay{k.gy, k.iy, Lx, 0}, ax{k.gx, k.ix, k.geo.Ly, cuty ? 6 * k.gy * Lx : 0};
    using Store = typename Par::Store;
    {
        const Store* src = static_cast<const Store*>(k.src);
        int x = xs, y = ys;
        for (int m = c; m < pairs; m += T) {
            const int X = k.x0 + x, Y = k.y0 + y, XB = k.x0 + bw - 1 - x, YB = k.y0 + bh - 1 - y;
            float va[9], vb[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                va[i] = (float)src[pull_at(k.geo, i, X, Y)];
                vb[i] = (float)src[pull_at(k.geo, i, XB, YB)];
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                cell[9 * m + i] = va[i];
                cell[9 * (nn - 1 - m) + i] = vb[i];
            }
            x += dx;
            y += dy;
            if (x >= bw) {
                x -= bw;
                ++y;
            }
        }
    }

    __syncthreads();

    // in bytes: a row of cells, all cells; the steps between a thread's pairs; the
    // steps so far modulo the block
    const uint32_t row = 36u * bw, all = row * bh, cell0 = smem_u32(cell);
    const uint32_t dxo = 36u * dx, dyo = row * dy, dnode = (uint32_t)dx + (uint32_t)Lx * (uint32_t)dy;
    const uint32_t node0 = (uint32_t)k.x0 + (uint32_t)Lx * (uint32_t)k.y0;
    const uint32_t nodes = 2u * node0 + (uint32_t)(bw - 1) + (uint32_t)Lx * (uint32_t)(bh - 1);   // A's plus B's
    uint32_t sx = 0, sy = 0;
    int until = k.first;             // next step to sample
    int nsum = 0;                    // sampled steps so far
    int funtil = k.fields ? k.ffirst : k.n, nfield = 0;
    bool pending = false;            // the previous step's partials wait in the slots
    for (int st = 0; st < k.n; ++st) {
        const uint32_t t = k.t0 + (uint32_t)st;
        const bool last = st == k.n - 1;
        const bool smp = SAMPLE != kResQuiet && st == until;
        if (smp) until = k.every > k.n - st ? k.n : st + k.every;
        if constexpr (SAMPLE != kResQuiet) {
            if (pending) res_reduce<SAMPLE>(slots + ((nsum - 1) & 1) * nw * kResSlot, red, nwork);
            pending = false;
        }
        float* fields = nullptr;
        if (st == funtil) {
            fields = k.fields + (size_t)nfield++ * 3 * Lx * k.geo.Ly;
            funtil = k.fevery > k.n - st ? k.n : st + k.fevery;
        }
        const uint64_t* in = k.mail + (size_t)(st & 1) * k.mail_words;
        uint64_t* out = k.mail + (size_t)((st + 1) & 1) * k.mail_words;
        // node A's column and row as byte offsets, and its number in the lattice
        uint32_t xo = 36u * xs, yo = row * ys, node = node0 + (uint32_t)xs + (uint32_t)Lx * (uint32_t)ys;
        for (int m0 = warp * 32; m0 < pairs; m0 += T) {
            const int m = m0 + lane_id;
            const bool inA = m < pairs, inB = inA && 2 * m != nn - 1;
            // the offsets less the steps so far, modulo the block (unsigned: the
            // one that has not wrapped is the smaller one)
            ResCells a;
            a.c[0] = cell0 + min(xo + sx, xo + sx - row);
            a.c[1] = cell0 + xo;
            a.c[2] = cell0 + min(xo - sx, xo - sx + row);
            a.r[0] = min(yo + sy, yo + sy - all);
            a.r[1] = yo;
            a.r[2] = min(yo - sy, yo - sy + all);
            a.kb = 2u * cell0 + all - 36u;
            const uint32_t nodeA = node, nodeB = nodes - node;
            // places in the lattice, where they are needed
            const auto place = [&](int& X, int& Y, int& XB, int& YB) {
                const int x = (int)(xo / 36u), y = (int)(yo / row);
                X = k.x0 + x;
                Y = k.y0 + y;
                XB = k.x0 + bw - 1 - x;
                YB = k.y0 + bh - 1 - y;
            };
            const ResEdge e{cutx && xo == 0, cutx && xo == row - 36u, cuty && yo == 0, cuty && yo == all - row};
            const bool edge = CUT && inA && e.any();
            if (edge && st > 0) {   // what comes across the cut: into this thread's own cells
                const uint32_t tag = k.tag0 + (uint32_t)st;
                int X, Y, XB, YB;
                place(X, Y, XB, YB);
                if (e.b) res_edge_in<1, 2, 5, 6>(in, tag, ay, X, XB, a, false, false, gave_up);
                if (e.t) res_edge_in<1, 4, 7, 8>(in, tag, ay, X, XB, a, false, false, gave_up);
                if (e.l) res_edge_in<0, 1, 5, 8>(in, tag, ax, Y, YB, a, e.b, e.t, gave_up);
                if (e.r) res_edge_in<0, 3, 7, 6>(in, tag, ax, Y, YB, a, e.t, e.b, gave_up);
            }
            auto load = [&](f2(&g)[9]) {
                if (inA) {
                    load_cells(a, g);
                } else {   // a lane past the end: any valid state
#pragma unroll
                    for (int i = 0; i < 9; ++i) g[i] = f2(1.f);
                }
            };
            f2 g[9];
            load(g);
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = par.decode(g[i], i);
            if (sizeof(Store) == 4 && fields) {
                f2 d[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) d[i] = g[i] - f2(par.ref(i));
                const f2 fr = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])) + d[8];
                const f2 fx = (d[1] - d[3]) + ((d[5] - d[6]) + (d[8] - d[7]));
                const f2 fy = (d[2] - d[4]) + ((d[5] + d[6]) - (d[7] + d[8]));
                const size_t N = (size_t)Lx * k.geo.Ly;
                int X, Y, XB, YB;
                place(X, Y, XB, YB);
                if (inA) {
                    float* o = fields + (size_t)Y * Lx + X;
                    o[0] = fr.v.x;
                    o[N] = fx.v.x;
                    o[2 * N] = fy.v.x;
                }
                if (inB) {
                    float* o = fields + (size_t)YB * Lx + XB;
                    o[0] = fr.v.y;
                    o[N] = fx.v.y;
                    o[2 * N] = fy.v.y;
                }
            }
            auto refetch = [&](f2* out9) {
                f2(&gg)[9] = *reinterpret_cast<f2(*)[9]>(out9);
                load(gg);
                if constexpr (SAMPLE != kResQuiet) {
                    if (smp) {
                        f2 h[9];
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            h[i] = par.scaled(gg[i], i);
                            if (!inB) h[i] = f2(inA ? h[i].v.x : 0.f, 0.f);
                        }
                        if constexpr (kExact)
                            prod_stage(gp, h);
                        else
                            gram_stage(gh, h);
                    }
                }
#pragma unroll
                for (int i = 0; i < 9; ++i) gg[i] = par.decode(gg[i], i);
            };
            f2 f[9];
            const uint32_t stt =
                collide_basis<f2, BASIS>(g, PairNoiseT<typename Par::Key>{par.key, nodeA, nodeB, t}, refetch, k.lut, par.cc, f);
            if (stt) {
                const unsigned long long at = (unsigned long long)st << 32;   // nodes are below 2^31
                if (inA && (stt & 0xFF)) atomicMin(first_error(), at | nodeA << 1 | ((stt & 0xFF) == kStatusNonfinite));
                if (inB && (stt >> 8)) atomicMin(first_error(), at | nodeB << 1 | ((stt >> 8) == kStatusNonfinite));
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = par.encode(f[i], i);
            if (last) {
                Store* dst = static_cast<Store*>(k.dst);
                int X, Y, XB, YB;
                place(X, Y, XB, YB);
                if (inA) store_lane(dst + at(k.geo, 0, X, Y), k.geo, X, Y, f, 0);
                if (inB) store_lane(dst + at(k.geo, 0, XB, YB), k.geo, XB, YB, f, 1);
            } else if (inA) {
                store_cells(a, f, inB);
                if (edge) {
                    const uint32_t tag = k.tag0 + (uint32_t)st + 1u;
                    int X, Y, XB, YB;
                    place(X, Y, XB, YB);
                    if (e.t) res_edge_out<1, 2, 5, 6>(out, tag, ay, X, XB, a, false, false, inB);
                    if (e.b) res_edge_out<1, 4, 7, 8>(out, tag, ay, X, XB, a, false, false, inB);
                    if (e.r) res_edge_out<0, 1, 5, 8>(out, tag, ax, Y, YB, a, e.t, e.b, inB);
                    if (e.l) res_edge_out<0, 3, 7, 6>(out, tag, ax, Y, YB, a, e.b, e.t, inB);
                }
            }
            // after the stores: what the neighbours wait for leaves first
            if constexpr (SAMPLE != kResQuiet) {
                if (smp) {
                    if constexpr (kExact)
                        prod_sums(gp, reinterpret_cast<float(&)[8]>(gc));
                    else
                        gram_mma(gh, reinterpret_cast<float(&)[8]>(gc));
                }
            }
            xo += dxo;
            yo += dyo;
            node += dnode;
            if (xo >= row) {
                xo -= row;
                yo += row;
                node += (uint32_t)(Lx - bw);
            }
        }
        if constexpr (SAMPLE != kResQuiet) {
            if (smp) {
                if (warp < nwork)
                    res_publish<SAMPLE>(reinterpret_cast<float(&)[8]>(gc), slots + ((nsum & 1) * nw + warp) * kResSlot);
                ++nsum;
                pending = true;
            }
        }
        sx = sx + 36u == row ? 0u : sx + 36u;
        sy = sy + row == all ? 0u : sy + row;
        if (!last) __syncthreads();
    }
    __syncthreads();
    if (c == 0) {
        const unsigned long long e = *first_error();
        if (e != ~0ull)
            record_earliest(k.err, e & 1 ? kStatusNonfinite : kStatusInvalidVelocity, (uint32_t)e >> 1,
                            k.t0 + (uint32_t)(e >> 32), k.t0, k.n);
        if (*gave_up) record_earliest(k.err, kStatusTimeout, -1, k.t0 + ((uint32_t)gave_up[1] - k.tag0), k.t0, k.n);
    }
    if constexpr (SAMPLE != kResQuiet) {
        if (pending) res_reduce<SAMPLE>(slots + ((nsum - 1) & 1) * nw * kResSlot, red, nwork);
        __syncthreads();
        if (nsum)
            for (int q = c; q < kSums; q += T) atomicAdd(&k.acc[q], res_sum<SAMPLE>(red, q, par.s));
    }
}

// A lattice in one block goes without the code of the edges, whose calls cost
// registers around them where they are never made: us per step with one body for
// both and with two: 21 x 21 2.12 / 1.99, 384 x 21^2 5.86 / 5.60, 1000 x 750 (cut)
// 15.16 / 15.03.
template <int BASIS, int SAMPLE, class Par>
__device__ __forceinline__ void resident_run(const ResBlock& k, const Par& par, unsigned char* smem) {
    if (k.gx * k.gy > 1)
        resident_run_of<BASIS, SAMPLE, true>(k, par, smem);
    else
        resident_run_of<BASIS, SAMPLE, false>(k, par, smem);
}

// One lattice (a handle): CTA b is block b of gx x gy.
struct ResidentArgs {
    ResBlock k;          // x0, y0, bw, bh, ix, iy are the CTA's own
    float ref[9];        // f^0(rho0, u0)
    float sinv;          // 1 / s
    float snref[9];      // -ref / s
    float scale;         // FP16 store: sqrt(kT)
    double s;            // scale of the staged deviations
};

// The block of column ix and row iy of the grid of blocks.
__host__ __device__ __forceinline__ void res_place(ResBlock& k, int ix, int iy) {
    k.ix = ix;
    k.iy = iy;
    k.x0 = (int)((long long)ix * k.geo.Lx / k.gx);
    k.y0 = (int)((long long)iy * k.geo.Ly / k.gy);
    k.bw = (int)((long long)(ix + 1) * k.geo.Lx / k.gx) - k.x0;
    k.bh = (int)((long long)(iy + 1) * k.geo.Ly / k.gy) - k.y0;
}

struct LatticePar {
    using Store = float;
    using Key = const NoiseKey&;
    const NoiseKey& key;
    const CollideConst<float>& cc;
    const ResidentArgs& a;
    double s;
    __device__ __forceinline__ f2 scaled(f2 f, int i) const { return mad(f, f2(a.sinv), f2(a.snref[i])); }
    __device__ __forceinline__ float ref(int i) const { return a.ref[i]; }
    __device__ __forceinline__ f2 decode(f2 v, int) const { return v; }
    __device__ __forceinline__ f2 encode(f2 f, int) const { return f; }
};

// The FP16 deviation store (flb_step_fp16.cu): stored values h = (f - c) / s, s =
// sqrt(kT), rounded to FP16 in every step.
struct LatticePar16 {
    using Store = __half;
    using Key = const NoiseKey&;
    const NoiseKey& key;
    const CollideConst<float>& cc;
    const ResidentArgs& a;
    double s;
    __device__ __forceinline__ f2 scaled(f2 v, int) const { return v * f2(a.scale); }
    __device__ __forceinline__ float ref(int i) const { return a.ref[i]; }
    __device__ __forceinline__ f2 decode(f2 v, int i) const { return mad(v, f2(a.scale), f2(a.ref[i])); }
    __device__ __forceinline__ f2 encode(f2 f, int i) const {
        const f2 h = mad(f, f2(a.sinv), f2(a.snref[i]));
        return f2(__half22float2(__floats2half2_rn(h.v.x, h.v.y)));
    }
};

template <int BASIS, int SAMPLE, class Par>
__global__ void __launch_bounds__(kResMaxWarps * 32, 1)
resident_kernel(const __grid_constant__ ResidentArgs a, const __grid_constant__ CollideConst<float> cc) {
    extern __shared__ __align__(128) unsigned char res_smem[];
    ResBlock k = a.k;
    const int iy = blockIdx.x / k.gx;
    res_place(k, blockIdx.x - iy * k.gx, iy);
    resident_run<BASIS, SAMPLE>(k, Par{cc.key, cc, a, a.s}, res_smem);
}

// Steps of one launch: without sampling at least kResMinSteps (fewer cost less one
// by one: 21 x 21 4.0 / 8.0 / 10.3 us for calls of 1, 2, 3 steps, the last in one
// launch). Sampled calls of one and two steps take 8.2 and 10.3 us (21 x 21), 8.2 and
// 12.3 (300 x 130), 24.6 and 41.1 (1000 x 750) against 6.8 and 13.5, 8.0 and 16.1, 20.8
// and 41.6 one by one.
constexpr int kResMinSteps = 3;
constexpr int kResMaxSteps = 1 << 20;

// Steps of the next launch, of n that are left, us (estimated) each: about 10 ms at
// most, for a launch holds its SMs to its end and other streams' kernels come in
// between launches only. (A launch of its own costs 3 to 6 us, below 0.1 % of that.)
// What is left is never too short for one more.
constexpr double kResLaunchUs = 10000;
inline int64_t resident_launch_steps(int64_t n, double us) {
    const int64_t most = us * kResMaxSteps > kResLaunchUs ? (int64_t)(kResLaunchUs / us) : kResMaxSteps;
    const int64_t m = most < 2 * kResMinSteps ? 2 * kResMinSteps : most;
    return n <= m ? n : (n - m < kResMinSteps ? m - kResMinSteps : m);
}

// A lattice's launch: how it is cut, and what the launch needs.
struct ResidentPlan {
    int gx = 0, gy = 0;      // 0: no resident launch
    int threads[2] = {0, 0};
    double us = 0;           // estimated time of a step without sampling
    size_t smem[2] = {0, 0}; // without, with sampling (0: does not fit)
    long long mail_words = 0;
};

constexpr size_t kResSmemMax = 227 * 1024;

// Estimated microseconds of a step of a block of bw x bh nodes, wp warp passes,
// of a lattice cut into gx x gy blocks.
double resident_step_us(int wp, int gx, int gy, int bw, int bh);
// Whether a launch of many steps is faster than one launch per step.
bool resident_pays(const ResidentPlan& p, double nodes, bool half, bool sample);
// Cut a lattice for the given number of SMs; `cut` = false: one block only.
ResidentPlan resident_plan(int Lx, int Ly, int sms, bool cut, bool half);
// Raise the kernels' dynamic shared memory limit (once per plan).
cudaError_t resident_prepare(const ResidentPlan& p, int basis, bool half);
cudaError_t resident_step(const ResidentPlan& p, const ResidentArgs& a, const CollideConst<float>& cc, int basis,
                          bool half, bool sample, cudaStream_t s);

}  // namespace flb
