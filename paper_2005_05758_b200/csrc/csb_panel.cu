// CSB product with one and with few vectors over the panel layout, fp32 accumulation (and the
// fixed-point product, csb_fixed.cu).
//
// The work of the paper's CSB-Engine (Section 4.3.1: read the kept inputs through ColIdx,
// multiply by the kernel matrix, accumulate into the outputs through RowIdx, sum along the
// block-row) is arranged so that the irregular parts happen once per CTA and the inner loop is
// a plain stream:
//
//   * a CTA owns a contiguous range of output rows and with it one panel: of every block with
//     kept rows in the range, those rows.  Every output is written by exactly one CTA, so
//     nothing is joined across CTAs and there are no atomics on y;
//   * one bulk copy brings in the panel's bookkeeping, one brings in x, and the kept inputs of
//     all of the panel's blocks are gathered once into shared memory;
//   * the panel's values flow through one shared-memory ring in fixed-size stages.  Whoever
//     finishes the last item of a stage refills its slot, so there is no producer thread and
//     nobody waits for a slower neighbour;
//   * a warp takes one bundle at a time: one item (up to 32 kept rows of a block) on all its
//     lanes, or two items of at most 16 rows / four of at most 8 rows side by side on lane
//     groups of 16 / 8, so that the fixed work per item is shared.  A lane owns one kept row
//     and reads 16 bytes = 8 kept columns per step; lanes left over in a group split the
//     columns 2-, 4-, ... ways and a few shuffles join them.  Products are accumulated with
//     packed fp32 multiply-adds;
//   * with two or four vectors a pass the same walk holds a sum per vector: a weight is read and
//     converted once, the gathered inputs of the vectors lie side by side;
//   * every warp adds into its own copy of the CTA's output rows; at the end the CTA adds the
//     copies in warp order and stores y.  The deal of items to warps is part of the plan, so
//     the result does not depend on timing.
//
// What bounds it: a matrix of a few MB, start-up and the latency of copies, gather and walk one behind
// the other (3072 x 1536 fp32 at 8x: one vector 3.6 us, four 5.2; the kernel of csb_product.cu 10.3 and 14.9,
// which walks block by block and joins its CTAs through global memory); a large one, bundles per warp
// (8192 x 8192 fp16 at 4x: 10.8 us for 33 MB).
#include <algorithm>
#include <cstdlib>

#include "csb_internal.hpp"
#include "csb_device.cuh"

namespace csb {

struct PanelArgs {
    const uint8_t* panels;
    const void* x;                     // float or int16 [nb, ldx]
    void* y;                           // float or int64 [nb, ldy]
    long long ldx, ldy;
    int nb;                            // batch columns of this pass, 1..BT
    uint32_t* status;
    int rows, cols;
    int log2_stage, log2_slots;        // ring = 2^log2_slots stages of 2^log2_stage bytes
    int max_rows;                      // accumulators per warp
    int max_xg, max_meta;
    int staged;                        // PanelPlan::staged
    uint4 cta[kMaxPanelCtas];          // PanelCta per CTA
#ifdef CSB_PANEL_CLOCKS
    unsigned long long* clocks;        // instrumented build only: [CTA][8] wall-clock stamps in ns
#endif
};

#ifdef CSB_PANEL_CLOCKS
#define PANEL_STAMP(i) do { if (threadIdx.x == 0) a.clocks[(size_t)blockIdx.x * 8 + (i)] = global_ns(); } while (0)
#else
#define PANEL_STAMP(i) do { } while (0)
#endif

__host__ __device__ inline size_t panel_align(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Shared-memory carve-up, identical on host and device: BT input vectors, BT gathered values per kept
// column, BT sums per row.  Float inputs: fp32 sums per warp; fixed point: int16 inputs, one 64-bit sum per CTA.
struct PanelSmem {
    size_t ring, xs, xs_row, xg, zs, meta, bars, done, issued, dead, total;
    __host__ __device__ PanelSmem(bool q16, bool staged, int BT, int W, int log2_stage, int log2_slots, int cols, int max_xg, int max_rows, int max_meta) {
        const int slots = 1 << log2_slots;
        ring = 0;
        xs = (size_t)slots << log2_stage;
        xs_row = panel_align((size_t)cols * (q16 ? 2 : 4), 16);
        xg = xs + (staged ? xs_row * BT : 0);
        zs = panel_align(xg + (size_t)max_xg * BT * (q16 ? 2 : 4), 16);
        meta = panel_align(zs + (size_t)max_rows * BT * (q16 ? 8 : 4 * W), 128);
        bars = panel_align(meta + (size_t)max_meta, 16);
        done = bars + (size_t)(slots + 2) * 8;
        issued = done + (size_t)slots * 4;
        dead = issued + (size_t)slots * 4;
        total = panel_align(dead + 4, 16);
    }
};

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
          "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 h2f2(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }

// Blocks until the grids this one depends on (the work in front of it on the stream) have
// completed and their writes are visible; returns at once for an ordinary launch.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Wait for a phase; gives up after the wall-clock bound or as soon as another warp of the CTA
// has given up.
__device__ __forceinline__ bool panel_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* dead) {
    if (mbar_try_wait(bar, parity)) return true;
    unsigned long long t0 = 0;                     // the clock is a slow read: looked at every 256 failed polls only
    unsigned int spins = 0;
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++spins & 255u) == 0) {
            if (*dead) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > kCopyWaitNs) return false;
        }
    }
}

// Wait until stage `st` of the value stream has landed in its ring slot.  The barrier of a slot
// is tested by phase parity, which can only tell apart two neighbouring phases: a warp that runs
// ahead and asks for the slot's next use while the copy of the current one is still in flight
// would be answered by the wrong phase.  So the warp first waits until the copy it needs has
// been issued (the slot's issue count, written by whoever refills it); from then on the barrier
// is either in that phase or just past it, and the parity test is exact.
__device__ __forceinline__ bool panel_wait_stage(uint64_t* full, volatile uint32_t* issued, uint32_t st, int log2_slots,
                                                 volatile uint32_t* dead) {
    const uint32_t slot = st & ((1u << log2_slots) - 1u), use = st >> log2_slots;
    if (use > 0u && issued[slot] <= use) {
        unsigned long long t0 = 0;
        unsigned int spins = 0;
        while (issued[slot] <= use) {
            if ((++spins & 255u) == 0) {
                if (*dead) return false;
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                else if (now - t0 > kCopyWaitNs) return false;
            }
        }
    }
    return panel_wait(&full[slot], use & 1u, dead);
}

// Two 16-bit weights times the signed / unsigned bytes 0, 1 (lo) or 2, 3 (hi) of b, added to c.
__device__ __forceinline__ int dp2a_lo_s(uint32_t w, uint32_t b, int c) { int d; asm("dp2a.lo.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(b), "r"(c)); return d; }
__device__ __forceinline__ int dp2a_hi_s(uint32_t w, uint32_t b, int c) { int d; asm("dp2a.hi.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(b), "r"(c)); return d; }
__device__ __forceinline__ int dp2a_lo_u(uint32_t w, uint32_t b, int c) { int d; asm("dp2a.lo.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(b), "r"(c)); return d; }
__device__ __forceinline__ int dp2a_hi_u(uint32_t w, uint32_t b, int c) { int d; asm("dp2a.hi.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(w), "r"(b), "r"(c)); return d; }

// The lane's share of one item in fixed point, added into the CTA's 64-bit sums.  An input is split
// into its signed high and unsigned low byte, x = 256 xh + xl, so that a pair of weights costs one
// dp2a per half and nothing is converted; the gathered inputs lie in quads of columns, per batch
// column four high bytes and four low bytes.  Neither 32-bit sum can overflow: an item has at most
// 128 columns, |w xh| <= 2^22 and |w xl| < 2^23, so the sums stay below 2^29 and 2^30.  Integer sums
// do not depend on their order, hence the shared-memory atomics.
template <int BT>
__device__ __forceinline__ void panel_item_q16(const uint8_t* ring, uint32_t ring_mask, uint32_t off, const uint2* __restrict__ xq4, int n, int m,
                                               int gl, int logp, int logg, int my_row, bool live, unsigned long long* zs) {
    int hi[BT], lo[BT];
#pragma unroll
    for (int b = 0; b < BT; ++b) { hi[b] = 0; lo[b] = 0; }
    const int r = gl & ((1 << logp) - 1), sub = gl >> logp, S = 32 >> (logg + logp);
    const int noct = n >> 3;
    uint32_t q = off + ((uint32_t)(sub * m + r) << 4);
    const uint32_t qstep = (uint32_t)(S * m) << 4;
    const uint2* xq = xq4 + (size_t)2 * sub * BT;
#pragma unroll 2
    for (int o = sub; o < noct; o += S) {
        const uint4 w = *reinterpret_cast<const uint4*>(ring + (q & ring_mask));
#pragma unroll
        for (int b = 0; b < BT; ++b) {
            const uint2 x0 = xq[b], x1 = xq[BT + b];
            hi[b] = dp2a_lo_s(w.x, x0.x, hi[b]); lo[b] = dp2a_lo_u(w.x, x0.y, lo[b]);
            hi[b] = dp2a_hi_s(w.y, x0.x, hi[b]); lo[b] = dp2a_hi_u(w.y, x0.y, lo[b]);
            hi[b] = dp2a_lo_s(w.z, x1.x, hi[b]); lo[b] = dp2a_lo_u(w.z, x1.y, lo[b]);
            hi[b] = dp2a_hi_s(w.w, x1.x, hi[b]); lo[b] = dp2a_hi_u(w.w, x1.y, lo[b]);
        }
        q += qstep;
        xq += 2 * S * BT;
    }
    if ((n & 7) && gl < m) {
        // the last n % 8 columns: [row][4], [row][2], [row][1] behind the octets
        uint32_t tb = off + ((uint32_t)(noct * m) << 4);
        const uint2* xt = xq4 + (size_t)2 * noct * BT;
        if (n & 4) {
            const uint2 w = *reinterpret_cast<const uint2*>(ring + ((tb + 8u * gl) & ring_mask));
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                const uint2 x0 = xt[b];
                hi[b] = dp2a_lo_s(w.x, x0.x, hi[b]); lo[b] = dp2a_lo_u(w.x, x0.y, lo[b]);
                hi[b] = dp2a_hi_s(w.y, x0.x, hi[b]); lo[b] = dp2a_hi_u(w.y, x0.y, lo[b]);
            }
            tb += 8u * m; xt += BT;
        }
        if (n & 2) {
            const uint32_t w = *reinterpret_cast<const uint32_t*>(ring + ((tb + 4u * gl) & ring_mask));
#pragma unroll
            for (int b = 0; b < BT; ++b) { hi[b] = dp2a_lo_s(w, xt[b].x, hi[b]); lo[b] = dp2a_lo_u(w, xt[b].y, lo[b]); }
            tb += 4u * m;
        }
        if (n & 1) {
            const uint32_t w = *reinterpret_cast<const uint16_t*>(ring + ((tb + 2u * gl) & ring_mask));   // upper weight 0
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                if (n & 2) { hi[b] = dp2a_hi_s(w, xt[b].x, hi[b]); lo[b] = dp2a_hi_u(w, xt[b].y, lo[b]); }
                else { hi[b] = dp2a_lo_s(w, xt[b].x, hi[b]); lo[b] = dp2a_lo_u(w, xt[b].y, lo[b]); }
            }
        }
    }
    // join the lanes that split the columns of a row
    const int pmin = logg ? (int)__reduce_min_sync(0xffffffffu, 1u << logp) : 1 << logp;
    for (int o = 16 >> logg; o >= pmin; o >>= 1)
#pragma unroll
        for (int b = 0; b < BT; ++b) {
            const int th = __shfl_xor_sync(0xffffffffu, hi[b], o), tl = __shfl_xor_sync(0xffffffffu, lo[b], o);
            if (o >= (1 << logp)) { hi[b] += th; lo[b] += tl; }
        }
    if (live)
#pragma unroll
        for (int b = 0; b < BT; ++b) {
            const long long v = ((long long)hi[b] << 8) + (long long)lo[b];
            if (v) atomicAdd(zs + (size_t)my_row * BT + b, (unsigned long long)v);
        }
}

// The lane's share of one item of fp16 or fp32 values with BT input vectors.  The gathered inputs lie in
// quads of columns, BT float4 to a quad; a weight is read and converted once for all vectors.
template <int VAL, int BT>
__device__ __forceinline__ void panel_item_float(const uint8_t* ring, uint32_t ring_mask, uint32_t off, const float4* __restrict__ xq4, int n, int m, int gl,
                                                 int logp, int logg, float (&acc)[BT]) {
    constexpr int U = VAL == CSB_F32 ? 4 : 8, Q = U / 4;   // columns and quads of 16 bytes
    float2 lo[BT], hi[BT];
#pragma unroll
    for (int b = 0; b < BT; ++b) { lo[b] = make_float2(0.f, 0.f); hi[b] = make_float2(0.f, 0.f); }
    const int r = gl & ((1 << logp) - 1), sub = gl >> logp, S = 32 >> (logg + logp);
    const int whole = n / U;
    uint32_t q = off + ((uint32_t)(sub * m + r) << 4);
    const uint32_t qstep = (uint32_t)(S * m) << 4;
    const float4* xq = xq4 + (size_t)Q * sub * BT;
#pragma unroll 2
    for (int o = sub; o < whole; o += S) {
        const uint4 w = *reinterpret_cast<const uint4*>(ring + (q & ring_mask));
        if (VAL == CSB_F32) {
            const float2 w0 = make_float2(__uint_as_float(w.x), __uint_as_float(w.y)), w1 = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                const float4 x = xq[b];
                lo[b] = ffma2(w0, make_float2(x.x, x.y), lo[b]);
                hi[b] = ffma2(w1, make_float2(x.z, x.w), hi[b]);
            }
        } else {
            const float2 w0 = h2f2(w.x), w1 = h2f2(w.y), w2 = h2f2(w.z), w3 = h2f2(w.w);
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                const float4 x = xq[b], y = xq[BT + b];
                lo[b] = ffma2(w0, make_float2(x.x, x.y), lo[b]);
                hi[b] = ffma2(w1, make_float2(x.z, x.w), hi[b]);
                lo[b] = ffma2(w2, make_float2(y.x, y.y), lo[b]);
                hi[b] = ffma2(w3, make_float2(y.z, y.w), hi[b]);
            }
        }
        q += qstep;
        xq += Q * S * BT;
    }
    if ((n & (U - 1)) && gl < m) {
        // the columns left over, by halves (csb_panel_plan.cpp); two of them and the last one lie in one quad
        uint32_t tb = off + ((uint32_t)(whole * m) << 4);
        const float* xt = reinterpret_cast<const float*>(xq4 + (size_t)Q * whole * BT);
        if (VAL != CSB_F32 && (n & 4)) {
            const uint2 w = *reinterpret_cast<const uint2*>(ring + ((tb + 8u * gl) & ring_mask));
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                const float4 x = *reinterpret_cast<const float4*>(xt + 4 * b);
                lo[b] = ffma2(h2f2(w.x), make_float2(x.x, x.y), lo[b]);
                hi[b] = ffma2(h2f2(w.y), make_float2(x.z, x.w), hi[b]);
            }
            tb += 8u * m; xt += 4 * BT;
        }
        if (n & 2) {
            float2 w;
            if (VAL == CSB_F32) { w = *reinterpret_cast<const float2*>(ring + ((tb + 8u * gl) & ring_mask)); tb += 8u * m; }
            else { w = h2f2(*reinterpret_cast<const uint32_t*>(ring + ((tb + 4u * gl) & ring_mask))); tb += 4u * m; }
#pragma unroll
            for (int b = 0; b < BT; ++b) lo[b] = ffma2(w, *reinterpret_cast<const float2*>(xt + 4 * b), lo[b]);
        }
        if (n & 1) {
            const float w = VAL == CSB_F32 ? *reinterpret_cast<const float*>(ring + ((tb + 4u * gl) & ring_mask))
                                           : __half2float(*reinterpret_cast<const __half*>(ring + ((tb + 2u * gl) & ring_mask)));
#pragma unroll
            for (int b = 0; b < BT; ++b) hi[b].x = fmaf(w, xt[4 * b + (n & 2)], hi[b].x);
        }
    }
#pragma unroll
    for (int b = 0; b < BT; ++b) acc[b] = (lo[b].x + hi[b].x) + (lo[b].y + hi[b].y);
}

// VAL: type of the values; fp16 and fp32 with fp32 inputs and outputs, 16-bit fixed point with 64-bit
// outputs.  BT: input vectors of a pass.
template <int VAL, int BT>
__global__ void __launch_bounds__(1024, 1) csb_panel_kernel(const __grid_constant__ PanelArgs a) {
    constexpr bool kQ = VAL == CSB_Q16;
    constexpr uint32_t kXBytes = kQ ? 2u : 4u;
    extern __shared__ __align__(128) uint8_t smem[];
    const int W = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool staged = BT == 1 || a.staged != 0;          // one vector always is
    const int nb = BT == 1 ? 1 : a.nb;
    const PanelSmem L(kQ, staged, BT, W, a.log2_stage, a.log2_slots, a.cols, a.max_xg, a.max_rows, a.max_meta);
    const uint4 ct = a.cta[blockIdx.x];
    const uint8_t* panel = a.panels + (size_t)ct.x * 16;
    const uint32_t meta_bytes = ct.y, value_bytes = ct.z;
    const uint8_t* values = panel + meta_bytes;
    const uint32_t slots = 1u << a.log2_slots, SB = 1u << a.log2_stage;
    const uint32_t ring_mask = (SB << a.log2_slots) - 1u;
    const uint32_t n_stages = (value_bytes + SB - 1u) >> a.log2_stage;
    uint8_t* ring = smem + L.ring;
    float* xs = reinterpret_cast<float*>(smem + L.xs);
    float* xg = reinterpret_cast<float*>(smem + L.xg);
    float* zs_all = reinterpret_cast<float*>(smem + L.zs);
    const uint8_t* meta = smem + L.meta;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.bars);
    uint64_t* metabar = full + slots;
    uint64_t* xbar = full + slots + 1;
    uint32_t* done = reinterpret_cast<uint32_t*>(smem + L.done);
    volatile uint32_t* issued = reinterpret_cast<volatile uint32_t*>(smem + L.issued);
    volatile uint32_t* s_dead = reinterpret_cast<volatile uint32_t*>(smem + L.dead);

    const bool x_bulk = staged && (reinterpret_cast<uintptr_t>(a.x) & 15) == 0 && (a.cols * kXBytes & 15) == 0 && (nb == 1 || (a.ldx * kXBytes & 15) == 0);
    // Launched with programmatic stream serialization, this grid may start while the kernel in
    // front of it on the stream is still draining: whatever comes next may be scheduled as early
    // as the hardware likes, and this grid touches x and y only behind grid_dependency_wait().
    // The panels are written once at plan time, so their copies go out before that wait.
    asm volatile("griddepcontrol.launch_dependents;");
    PANEL_STAMP(0);
    // the first copies go out from separate lanes of warp 0, each with the barrier it set up itself:
    // lane s < slots takes stage s, the next two lanes take the bookkeeping and x
    if (warp == 0 && (uint32_t)lane < slots + 2u) {
        const uint32_t s = (uint32_t)lane;
        mbar_init(&full[s], 1);
        if (s < slots) { done[s] = 0u; issued[s] = 0u; }
        if (s == slots) *s_dead = 0u;
        mbar_fence_init();
        // the bookkeeping first, then x (the gather of the inputs, which everything else waits for, needs
        // both; x may still be being written by the kernel in front), then the values
        if (s == slots) {
            mbar_expect_tx(metabar, meta_bytes);
            bulk_g2s(smem + L.meta, panel, meta_bytes, metabar);
        }
        if (s == slots + 1u && x_bulk) {
            grid_dependency_wait();
            const uint32_t xb = (uint32_t)a.cols * kXBytes;
            mbar_expect_tx(xbar, xb * (uint32_t)nb);
            for (int b = 0; b < nb; ++b)
                for (uint32_t off = 0; off < xb; off += 16384u)
                    bulk_g2s(smem + L.xs + b * L.xs_row + off, reinterpret_cast<const uint8_t*>(a.x) + (size_t)b * a.ldx * kXBytes + off, min(16384u, xb - off), xbar);
        }
        __syncwarp(slots + 2u >= 32u ? 0xffffffffu : (1u << (slots + 2u)) - 1u);
        if (s < slots && s < n_stages) {
            const uint32_t bytes = min(SB, value_bytes - (s << a.log2_stage));
            issued[s] = 1u;
            mbar_expect_tx(&full[s], bytes);
            bulk_g2s(ring + ((size_t)s << a.log2_stage), values + ((size_t)s << a.log2_stage), bytes, &full[s]);
        }
    }
    for (int i = threadIdx.x; i < (kQ ? 2 : W) * BT * a.max_rows; i += blockDim.x) zs_all[i] = 0.f;
    if (!x_bulk) {
        grid_dependency_wait();
        for (int b = 0; b < (staged ? nb : 0); ++b)
            for (int i = threadIdx.x; i < a.cols; i += blockDim.x) {
                if (kQ) reinterpret_cast<int16_t*>(smem + L.xs + b * L.xs_row)[i] = __ldg(reinterpret_cast<const int16_t*>(a.x) + (long long)b * a.ldx + i);
                else reinterpret_cast<float*>(smem + L.xs + b * L.xs_row)[i] = __ldg(reinterpret_cast<const float*>(a.x) + (long long)b * a.ldx + i);
            }
    }
    __syncthreads();                                       // barriers initialised, counters and sums cleared
    PANEL_STAMP(1);

    bool gave_up = !panel_wait(metabar, 0, s_dead);
    if (!gave_up && x_bulk) gave_up = !panel_wait(xbar, 0, s_dead);
    if (gave_up) *s_dead = 1u;
    gave_up = __syncthreads_or(gave_up) != 0;

    const PanelHeader* H = reinterpret_cast<const PanelHeader*>(meta);
    PANEL_STAMP(2);
    if (!gave_up) {
        // ---- gather the kept inputs of every block of the panel, once: four blocks per warp and
        // round, eight lanes per block, a lane resolves four column indices at a time (indices and
        // gathered inputs of a block are padded to four; padding indices are zero, i.e. the block's
        // first column, which exists)
        {
            const uint2* gath = reinterpret_cast<const uint2*>(meta + H->gather_off);
            const uint8_t* cidx = meta + H->cidx_off;
            const int n_gather = (int)H->n_gather;
            for (int g0 = warp * 4; g0 < n_gather; g0 += W * 4) {
                const int g = g0 + (lane >> 3);
                const uint2 gd = g < n_gather ? gath[g] : make_uint2(0u, 0u);
                const uint32_t xbase = gd.x & 0xffffu, n = gd.x >> 16, xoff = gd.y;
                for (uint32_t k = (uint32_t)(lane & 7) * 4u; k < n; k += 32u) {
                    const uint32_t c4 = *reinterpret_cast<const uint32_t*>(cidx + xoff + k);
                    if (kQ) {
                        const int16_t* xr = reinterpret_cast<const int16_t*>(xs) + xbase;
                        uint2* dst = reinterpret_cast<uint2*>(xg) + (size_t)((xoff + k) >> 2) * BT;
#pragma unroll
                        for (int b = 0; b < BT; ++b) {
                            // two inputs to a word, then the bytes sorted into high and low ones; a column past nb stays 0
                            uint2 h = make_uint2(0u, 0u);
                            if (b < nb) {
                                const uint32_t v0 = (uint16_t)xr[c4 & 0xffu], v1 = (uint16_t)xr[(c4 >> 8) & 0xffu];
                                const uint32_t v2 = (uint16_t)xr[(c4 >> 16) & 0xffu], v3 = (uint16_t)xr[c4 >> 24];
                                const uint32_t p0 = v0 | (v1 << 16), p1 = v2 | (v3 << 16);
                                h = make_uint2(__byte_perm(p0, p1, 0x7531), __byte_perm(p0, p1, 0x6420));
                            }
                            dst[b] = h;
                            xr += L.xs_row >> 1;
                        }
                        continue;
                    }
                    float4* dst = reinterpret_cast<float4*>(xg) + (size_t)((xoff + k) >> 2) * BT;
                    auto pick = [&](const float* xr, long long pitch) {
#pragma unroll
                        for (int b = 0; b < BT; ++b) {
                            // (a column past nb stays 0)
                            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (b < nb) v = make_float4(xr[c4 & 0xffu], xr[(c4 >> 8) & 0xffu], xr[(c4 >> 16) & 0xffu], xr[c4 >> 24]);
                            dst[b] = v;
                            xr += pitch;
                        }
                    };
                    if (staged) pick(xs + xbase, (long long)(L.xs_row >> 2));
                    else pick(reinterpret_cast<const float*>(a.x) + xbase, a.ldx);
                }
            }
        }
        __syncthreads();
        PANEL_STAMP(3);

        // ---- this warp's bundles: one item on all 32 lanes, or two / four small ones side by side
        const uint16_t* wb = reinterpret_cast<const uint16_t*>(meta + H->warp_off);
        const uint16_t* wlist = reinterpret_cast<const uint16_t*>(meta + H->list_off);
        const uint4* items = reinterpret_cast<const uint4*>(meta + H->items_off);
        const uint16_t* expect = reinterpret_cast<const uint16_t*>(meta + H->expect_off);
        const uint8_t* ridx = meta + H->ridx_off;
        const float4* xg4 = reinterpret_cast<const float4*>(xg);
        float* zs = zs_all + (size_t)warp * a.max_rows * BT;
        const uint32_t i_end = wb[warp + 1];
        uint32_t idx = wb[warp];
        uint32_t e = idx < i_end ? wlist[idx] : 0u;
        for (; idx < i_end; ++idx) {
            const int logg = (int)(e >> 14);
            const int gl = lane & ((32 >> logg) - 1), grp = lane >> (5 - logg);
            const uint4 d = items[(e & 0x3fffu) + grp];
            if (idx + 1 < i_end) e = wlist[idx + 1];          // on its way while this bundle is worked on
            const uint32_t off = d.x << 4;
            const uint32_t xoff4 = d.y & 0xffffu, roff = d.z & 0xffffu;
            const int zoff = (int)(int16_t)(d.y >> 16);
            const int m = (int)((d.z >> 16) & 0xffu), logp = (int)(d.z >> 24), n = (int)(d.w & 0xffffu);
            const int my_row = zoff + (int)ridx[roff + (gl < m ? gl : 0)];
            const uint32_t st = off >> a.log2_stage;          // the same for every member of the bundle
            if (__any_sync(0xffffffffu, !panel_wait_stage(full, issued, st, a.log2_slots, s_dead))) { *s_dead = 1u; break; }

            if (kQ) {
                panel_item_q16<BT>(ring, ring_mask, off, reinterpret_cast<const uint2*>(xg) + (size_t)xoff4 * BT, n, m, gl, logp, logg, my_row, gl < m,
                                   reinterpret_cast<unsigned long long*>(zs_all));
            } else if (VAL == CSB_F32 || BT > 1) {
                float acc[BT];
                panel_item_float<VAL, BT>(ring, ring_mask, off, xg4 + (size_t)xoff4 * BT, n, m, gl, logp, logg, acc);
                // join the lanes that split the columns of a row (fixed tree inside the lane group)
                const int pmin = logg ? (int)__reduce_min_sync(0xffffffffu, 1u << logp) : 1 << logp;
                for (int o = 16 >> logg; o >= pmin; o >>= 1)
#pragma unroll
                    for (int b = 0; b < BT; ++b) {
                        const float t = __shfl_xor_sync(0xffffffffu, acc[b], o);
                        if (o >= (1 << logp)) acc[b] += t;
                    }
                // members of a bundle may add into the same output: one lane group at a time
                for (int g = 0; g < (1 << logg); ++g) {
                    if (grp == g && gl < m)
#pragma unroll
                        for (int b = 0; b < BT; ++b) zs[my_row * BT + b] += acc[b];
                    __syncwarp();
                }
            } else {
            const int r = gl & ((1 << logp) - 1), sub = gl >> logp, S = 32 >> (logg + logp);
            const int noct = n >> 3;
            float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
            float2 b0 = make_float2(0.f, 0.f), b1 = make_float2(0.f, 0.f);
            {
                uint32_t q = off + ((uint32_t)(sub * m + r) << 4);
                const uint32_t qstep = (uint32_t)(S * m) << 4;
                const float4* xq = xg4 + xoff4 + 2 * sub;
                int o = sub;
                for (; o + S < noct; o += 2 * S) {          // two octets per round, loads first
                    const uint4 w = *reinterpret_cast<const uint4*>(ring + (q & ring_mask));
                    const uint4 v = *reinterpret_cast<const uint4*>(ring + ((q + qstep) & ring_mask));
                    const float4 x0 = xq[0], x1 = xq[1], x2 = xq[2 * S], x3 = xq[2 * S + 1];
                    a0 = ffma2(h2f2(w.x), make_float2(x0.x, x0.y), a0);
                    a1 = ffma2(h2f2(w.y), make_float2(x0.z, x0.w), a1);
                    b0 = ffma2(h2f2(v.x), make_float2(x2.x, x2.y), b0);
                    b1 = ffma2(h2f2(v.y), make_float2(x2.z, x2.w), b1);
                    a0 = ffma2(h2f2(w.z), make_float2(x1.x, x1.y), a0);
                    a1 = ffma2(h2f2(w.w), make_float2(x1.z, x1.w), a1);
                    b0 = ffma2(h2f2(v.z), make_float2(x3.x, x3.y), b0);
                    b1 = ffma2(h2f2(v.w), make_float2(x3.z, x3.w), b1);
                    q += 2 * qstep;
                    xq += 4 * S;
                }
                if (o < noct) {
                    const uint4 w = *reinterpret_cast<const uint4*>(ring + (q & ring_mask));
                    const float4 x0 = xq[0], x1 = xq[1];
                    a0 = ffma2(h2f2(w.x), make_float2(x0.x, x0.y), a0);
                    a1 = ffma2(h2f2(w.y), make_float2(x0.z, x0.w), a1);
                    a0 = ffma2(h2f2(w.z), make_float2(x1.x, x1.y), a0);
                    a1 = ffma2(h2f2(w.w), make_float2(x1.z, x1.w), a1);
                }
            }
            float acc = 0.f;
            if ((n & 7) && gl < m) {
                // the last n % 8 columns: [row][4], [row][2], [row][1] behind the octets
                uint32_t tb = off + ((uint32_t)(noct * m) << 4);
                const float* xt = xg + 4 * xoff4 + 8 * noct;
                if (n & 4) {
                    const uint2 w = *reinterpret_cast<const uint2*>(ring + ((tb + 8u * gl) & ring_mask));
                    const float4 x0 = *reinterpret_cast<const float4*>(xt);
                    b0 = ffma2(h2f2(w.x), make_float2(x0.x, x0.y), b0);
                    b1 = ffma2(h2f2(w.y), make_float2(x0.z, x0.w), b1);
                    tb += 8u * m; xt += 4;
                }
                if (n & 2) {
                    const uint32_t w = *reinterpret_cast<const uint32_t*>(ring + ((tb + 4u * gl) & ring_mask));
                    const float2 x0 = *reinterpret_cast<const float2*>(xt);
                    a0 = ffma2(h2f2(w), x0, a0);
                    tb += 4u * m; xt += 2;
                }
                if (n & 1) {
                    const __half w = *reinterpret_cast<const __half*>(ring + ((tb + 2u * gl) & ring_mask));
                    acc = __half2float(w) * xt[0];
                }
            }
            acc += ((a0.x + a1.x) + (b0.x + b1.x)) + ((a0.y + a1.y) + (b0.y + b1.y));
            // join the lanes that split the columns of a row (fixed tree inside the lane group)
            if (logg == 0) {
                for (int o = 16; o >= (1 << logp); o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane < m) zs[my_row] += acc;
            } else {
                const int pmin = (int)__reduce_min_sync(0xffffffffu, 1u << logp);
                for (int o = 16 >> logg; o >= pmin; o >>= 1) {
                    const float t = __shfl_xor_sync(0xffffffffu, acc, o);
                    if (o >= (1 << logp)) acc += t;
                }
                // members of a bundle may add into the same output: one lane group at a time
                for (int g = 0; g < (1 << logg); ++g) {
                    if (grp == g && gl < m) zs[my_row] += acc;
                    __syncwarp();
                }
            }
            }
            __syncwarp();
            // ---- the bundle is done with its stage; the last one out refills the slot
            if (lane == 0) {
                __threadfence_block();
                const uint32_t slot = st & (slots - 1u);
                if (atomicAdd(&done[slot], 1u) + 1u == (uint32_t)expect[st]) {
                    *reinterpret_cast<volatile uint32_t*>(&done[slot]) = 0u;
                    const uint32_t nx = st + slots;
                    if (nx < n_stages) {
                        __threadfence_block();
                        fence_proxy_async_all();
                        const uint32_t bytes = min(SB, value_bytes - (nx << a.log2_stage));
                        issued[slot] = issued[slot] + 1u;
                        mbar_expect_tx(&full[slot], bytes);
                        bulk_g2s(ring + ((size_t)slot << a.log2_stage), values + ((size_t)nx << a.log2_stage), bytes, &full[slot]);
                    }
                }
            }
        }
    }
#ifdef CSB_PANEL_CLOCKS
    if (lane == 0 && warp == 0) a.clocks[(size_t)blockIdx.x * 8 + 6] = global_ns();   // warp 0 out of its items
#endif
    __syncthreads();
    PANEL_STAMP(4);
    if (*s_dead) {
        // report, give the copies still in flight a bounded chance to land, and leave
        if (threadIdx.x == 0) {
            *(volatile uint32_t*)a.status = (uint32_t)kDevCopyTimeout;
            mbar_wait_bounded(metabar, 0);
            if (x_bulk) mbar_wait_bounded(xbar, 0);
            for (uint32_t s = 0; s < slots; ++s)
                if (issued[s]) mbar_wait_bounded(&full[s], (issued[s] - 1u) & 1u);
        }
        return;
    }

    // ---- add the warps' copies in warp order and store the CTA's rows
    const int n_rows = (int)H->n_rows, row0 = (int)H->row0;
    if (kQ) {
        for (int t = threadIdx.x; t < n_rows * nb; t += blockDim.x) {
            const int b = t / n_rows, r = t - b * n_rows;
            reinterpret_cast<long long*>(a.y)[(long long)b * a.ldy + row0 + r] = reinterpret_cast<const long long*>(zs_all)[r * BT + b];
        }
        return;
    }
    for (int t = threadIdx.x; t < n_rows * nb; t += blockDim.x) {
        const int b = BT == 1 ? 0 : t / n_rows, r = t - b * n_rows;
        float v = 0.f;
        for (int w = 0; w < W; ++w) v += zs_all[((size_t)w * a.max_rows + r) * BT + b];
        reinterpret_cast<float*>(a.y)[(long long)b * a.ldy + row0 + r] = v;
    }
    PANEL_STAMP(5);
    PANEL_STAMP(7);
}

#define CSB_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            set_error("%s failed: %s", #call, cudaGetErrorString(e_));                     \
            return e_ == cudaErrorMemoryAllocation ? CSB_ERR_ALLOC : CSB_ERR_CUDA;         \
        }                                                                                  \
    } while (0)

static int env_int(const char* name, int dflt) {
    const char* v = getenv(name);
    return v && *v ? atoi(v) : dflt;
}
static int log2_floor(int v) { int l = 0; while ((2 << l) <= v) ++l; return l; }

typedef void (*PanelKernel)(PanelArgs);
template <int VAL>
static PanelKernel pick_panel_kernel(int v) { return v == 0 ? csb_panel_kernel<VAL, 1> : v == 1 ? csb_panel_kernel<VAL, 2> : csb_panel_kernel<VAL, 4>; }
static PanelKernel panel_kernel(int val_dtype, int v) {
    return val_dtype == CSB_F16 ? pick_panel_kernel<CSB_F16>(v) : val_dtype == CSB_F32 ? pick_panel_kernel<CSB_F32>(v) : pick_panel_kernel<CSB_Q16>(v);
}

static int panel_stage() { return 1 << std::min(15, std::max(13, log2_floor(env_int("CSB_PANEL_STAGE", 16384)))); }

int plan_panels(const csb_matrix* A, PanelHostPlan* out) {
    if (env_int("CSB_NO_PANEL", 0)) return 1;
    const int warps = std::min(32, std::max(1, env_int("CSB_PANEL_WARPS", 32)));
    const int ctas = std::min<int>(kMaxPanelCtas, A->opts.ctas > 0 ? A->opts.ctas : A->sm_count);
    return plan_panels_host(A, ctas, warps, panel_stage(), 16384, 8192 / warps, out);
}

int upload_panels(csb_matrix* A, const PanelHostPlan& H) {
    const int warps = H.warps, stage = H.stage_bytes;
    PanelPlan* P = new PanelPlan();
    P->ctas = (int)H.cta.size(); P->warps = warps; P->stage_bytes = stage;
    P->max_xg = (int)H.max_xg; P->max_meta = (int)H.max_meta; P->max_rows = (int)std::max<size_t>(H.max_rows, 1);
    const int want_ring = std::min(17, std::max(log2_floor(stage) + 1, env_int("CSB_PANEL_RING_LOG2", 17)));
    // The deepest ring that leaves room for the rest, per variant of the kernel.  Several float vectors: not
    // below 64 KB (a pass of two over 8192 x 8192 fp32 values at 4x took 36 us on a ring of 32 KB, two passes of
    // one 26); where the vectors themselves are in its way, they stay in global memory and the gather reads
    // them there.
    const bool q16 = A->val_dtype == CSB_Q16;
    for (int v = 0; v < PanelPlan::kVariants; ++v)
        for (int direct = 0; direct < (q16 || v == 0 ? 1 : 2) && !P->log2_ring[v]; ++direct)
            for (int lr = want_ring; lr > log2_floor(stage); --lr) {
                if (v > 0 && !q16 && lr < std::min(16, want_ring)) break;
                const PanelSmem L(q16, !direct, PanelPlan::bt(v), warps, log2_floor(stage), lr - log2_floor(stage), (int)A->cols, P->max_xg, P->max_rows, P->max_meta);
                if (L.total <= A->smem_optin) { P->log2_ring[v] = lr; P->smem_bytes[v] = L.total; P->staged[v] = !direct; break; }
            }
    // the variant that takes one vector does not fit: the other path serves this matrix
    if (!P->log2_ring[0]) { delete P; return CSB_OK; }
    int prev = 0;
    CSB_CUDA(cudaGetDevice(&prev));
    CSB_CUDA(cudaSetDevice(A->device));
    A->panel = P;                                          // from here on csb_free releases what was allocated
    P->cta = H.cta;
    P->stream_bytes = (int64_t)H.bytes.size();
    P->balance = H.balance; P->warp_balance = H.warp_balance;
    CSB_CUDA(cudaMalloc((void**)&P->d_panels, std::max<size_t>(H.bytes.size(), 16)));
    CSB_CUDA(cudaMemcpy(P->d_panels, H.bytes.data(), H.bytes.size(), cudaMemcpyHostToDevice));
    for (int v = 0; v < PanelPlan::kVariants; ++v)
        CSB_CUDA(cudaFuncSetAttribute((const void*)panel_kernel(A->val_dtype, v), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A->smem_optin));
    CSB_CUDA(cudaDeviceSynchronize());
    CSB_CUDA(cudaSetDevice(prev));
    P->built = true;
    return CSB_OK;
}

void free_panels(csb_matrix* A) {
    PanelPlan* P = A->panel;
    if (!P) return;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(A->device);
    cudaFree(P->d_panels);
    cudaSetDevice(prev);
    delete P;
    A->panel = nullptr;
}

#ifdef CSB_PANEL_CLOCKS
static unsigned long long* g_panel_clocks = nullptr;
extern "C" int csb_debug_panel_clocks(unsigned long long* host_out, int ctas) {
    return (int)cudaMemcpy(host_out, g_panel_clocks, (size_t)ctas * 8 * 8, cudaMemcpyDeviceToHost);
}
#endif

static int launch_variant(const csb_matrix* A, int v, const void* x, int64_t ldx, int nb, void* y, int64_t ldy, void* stream) {
    const PanelPlan& P = *A->panel;
    const ProductPlan& Q = A->product;
    if (Q.h_status && *Q.h_status != 0) { set_error("an earlier product on this handle gave up waiting on the device (code %u)", *Q.h_status); return CSB_ERR_TIMEOUT; }
    int prev = 0;
    CSB_CUDA(cudaGetDevice(&prev));
    if (prev != A->device) CSB_CUDA(cudaSetDevice(A->device));
    PanelArgs a{};
    a.panels = P.d_panels; a.x = x; a.y = y; a.ldx = ldx; a.ldy = ldy; a.nb = nb; a.status = Q.d_status;
    a.rows = (int)A->rows; a.cols = (int)A->cols;
    a.log2_stage = log2_floor(P.stage_bytes); a.log2_slots = P.log2_ring[v] - a.log2_stage;
    a.staged = P.staged[v]; a.max_rows = P.max_rows; a.max_xg = P.max_xg; a.max_meta = P.max_meta;
    for (int c = 0; c < P.ctas; ++c) a.cta[c] = make_uint4(P.cta[c].off16, P.cta[c].meta_bytes, P.cta[c].value_bytes, P.cta[c].n_rows);
#ifdef CSB_PANEL_CLOCKS
    static unsigned long long* d_clocks = nullptr;
    if (!d_clocks) cudaMalloc((void**)&d_clocks, (size_t)kMaxPanelCtas * 8 * 8);
    a.clocks = d_clocks;
    g_panel_clocks = d_clocks;
#endif
    // Programmatic stream serialization lets this grid's start-up (barriers, first copies of the
    // panels) overlap the end of the kernel in front of it; the kernel orders itself behind that
    // kernel before it touches x or y.  CSB_PANEL_PDL=0 asks for an ordinary launch.
    const int use_pdl = env_int("CSB_PANEL_PDL", 1);      // read at every launch, so a caller can compare both kinds
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)P.ctas); cfg.blockDim = dim3((unsigned)P.warps * 32u);
    cfg.dynamicSmemBytes = P.smem_bytes[v]; cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = use_pdl ? 1u : 0u;
    cudaError_t e = cudaLaunchKernelEx(&cfg, panel_kernel(A->val_dtype, v), a);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (prev != A->device) cudaSetDevice(prev);
    if (e != cudaSuccess) { set_error("panel kernel launch failed: %s", cudaGetErrorString(e)); return CSB_ERR_CUDA; }
    return CSB_OK;
}

// Passes of as many vectors as are left and as leave room for a ring.
static int next_pass(const csb_matrix* A, int left) {
    int v = left >= 3 ? 2 : left - 1;
    while (v > 0 && !A->panel->log2_ring[v]) --v;
    return v;
}
// The other kernel (csb_product.cu) takes vectors in passes of four, two and one.  A pass of this one takes about
// half as long as one of its passes of four (3072 x 1536 fp32 values at 8x, four vectors: 5.0 against 14.9 us;
// 2048 x 8192 fp16, two vectors: 9.4 against 16.5), so up to twice as many are allowed.
bool panels_applicable(const csb_matrix* A, int batch) {
    if (!A->panel || !A->panel->built || A->val_dtype == CSB_Q16) return false;
    if (batch == 1) return true;
    if (batch > 8) return false;
    int passes = 0;
    for (int b = 0; b < batch; ++passes) b += std::min(batch - b, PanelPlan::bt(next_pass(A, batch - b)));
    return passes <= (batch <= 4 ? 1 : batch <= 6 ? 2 : 3);
}

template <typename X, typename Y>
static int launch_passes(const csb_matrix* A, const X* x, int64_t ldx, int batch, Y* y, int64_t ldy, void* stream) {
    for (int b0 = 0; b0 < batch;) {
        const int v = next_pass(A, batch - b0);
        const int nb = std::min(batch - b0, PanelPlan::bt(v));
        const int rc = launch_variant(A, v, x + (int64_t)b0 * ldx, ldx, nb, y + (int64_t)b0 * ldy, ldy, stream);
        if (rc != CSB_OK) return rc;
        b0 += nb;
    }
    return CSB_OK;
}

int launch_panels(const csb_matrix* A, const float* X, int64_t ldx, int batch, float* Y, int64_t ldy, void* stream) {
    return launch_passes(A, X, ldx, batch, Y, ldy, stream);
}

int launch_panels_q16(const csb_matrix* A, const int16_t* Xq, int64_t ldx, int batch, int64_t* acc, int64_t ldy, void* stream) {
    return launch_passes(A, Xq, ldx, batch, acc, ldy, stream);
}

}  // namespace csb
