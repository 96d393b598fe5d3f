// Batched CSB product on tcgen05 tensor cores, alone and as the time loop of a recurrent stack (fp16 values, fp32
// accumulation).
//
// The kernel matrices of the blocks (Section 4.3.1) are small and all different, and with rows and columns put back in their
// places a block is mostly zeros.  Tensor instructions for those zeros are cheap on this chip (8192 x 8192 dense, 64 columns as
// hi and lo halves: 10.5 us at the measured rate), so a warp expands the kept values into the dense tile and the contraction is a dense one:
//
//   * sixteen warps expand: lane = output row, eight 16-byte loads of its row's 64 columns, zeros where the row is not
//     kept, and one tcgen05.st puts the 32 words into TMEM as the A operand (128 rows x 64 columns per tile-window).  A never
//     passes through shared memory in its dense form, whose bandwidth the B operand needs;
//   * the inputs are packed into binary16 pairs x = hi + lo (no input precision is lost as long as |x| < 65504) as 128-byte
//     swizzled, K-major operand images, 64 columns each, the hi rows of all batch columns, then the lo rows; a
//     bulk copy brings an image as it is.  An input that binary16 cannot hold (NaN, infinite, from 65520 on) would make
//     NaN of its column's zeros too: it is left out of the product, marked, and where there is a mark the sums of
//     the rows that keep its column are set to NaN behind the product (spoil_sums);
//   * one warp issues the tcgen05.mma, one thread the copies of the inputs, one those of the values;
//   * the tensor cores add into TMEM with truncation, so the hi rows' sums of a unit (a tile over `flush` windows) start
//     from zero and are taken out by the same sixteen warps, which add them in registers with rounding.  The units' buffers
//     go round, so that the next ones run meanwhile.  The lo rows' sums are 2^-11 of the others and may stay until the end;
//   * a row group's column ranges are one thread-block cluster and are added in range order through distributed
//     shared memory: results are bit-reproducible, no scratch, no atomics.
//
// As a time loop (MODE 1 LSTM, 2 GRU) the grid stays for the whole sequence, each CTA with its tiles of one layer, whose
// quadrants are the gates of the same 32 hidden units.  In tick k layer l does step k - l.  After the cluster's sums every CTA does the
// gate arithmetic of its share of (units, batch column) and writes h_t into the other one of two buffers of operand
// images; a counter in global memory says when all CTAs have.  Only the thread that copies the inputs waits for it: the
// values of the next step are on their way and the first tiles expanded by then.
#pragma once

#include "csb_umma.hpp"
#include "csb_device.cuh"
#include "csb_gates.cuh"

namespace csb {

constexpr int kASlots = 8;                     // tile-windows of the A operand in TMEM, 32 columns each: two rounds
constexpr int kDCols = 256;                    // columns of TMEM for sums
constexpr uint32_t kNever = 0x40000000u;       // more arrivals than a sequence has
constexpr int kMaxXDepth = 4, kWRounds = 6;    // stages of inputs, rounds of values in shared memory
constexpr int kExpandThreads = kUmmaExpandWarps * 32, kUmmaThreads = kExpandThreads + 4 * 32;
// Windows of a stage of inputs: a round's, or half of it for 64 batch columns on one tile (32 KB).
__host__ __device__ constexpr int x_windows(int NB, int MT) { return MT == 2 || NB == 64 ? 2 : 4; }

struct UmmaPart {
    const uint8_t* stream;
    const UmmaCta* ctas;
    const UmmaRound* rounds;
    const UmmaQuad* quads;
    uint8_t* xp;               // packed inputs: per window an image of 2 * NB rows of 128 bytes (time loop: two such buffers)
    uint32_t* bad;             // NB / 4 words per window: are there marks in it?  (time loop: 16 bytes a buffer, the call and tick of the latest mark)
    float* Y;
    int cta_end;               // the part's CTAs end here in the grid
    int block_r, seg_words, windows;
};
struct UmmaArgs {
    UmmaPart part[kMaxLayers];
    long long ldy;
    uint32_t* status;
    int n_parts, nb, S, flush;
    int x_depth, w_bytes;                                  // stages of inputs, bytes for rounds of values (UmmaSmem)
    // time loop: a part is a layer
    const float* x; float* y; const float* state0;        // [T, nb, in_size[0]]; [T, nb, H] or null; [L, nb, H]: c (LSTM) or h (GRU) at the start
    float *hT, *cT;                                        // [L, nb, H] or null
    const float* bias[kMaxLayers];
    int in_size[kMaxLayers];
    uint32_t* count;                                       // CTAs that have finished a tick, summed over ticks
    unsigned long long limit_ns;
    uint32_t never;                                        // test hook: arrivals that never come,
    int never_step;                                        // and the step at which they are missing for the warps that pack x alone
    int T, H, x_vec;                                       // x_vec: rows of x start at multiples of 16 bytes
    uint32_t call;                                         // this call's number
};

// ---- tcgen05 -----------------------------------------------------------------------------------------
__device__ __forceinline__ void tc_alloc(uint32_t smem_out, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_out), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols));
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D (TMEM) (+)= A (TMEM, 128 x 16 binary16) . B (shared memory, K-major)
__device__ __forceinline__ void tc_mma_f16(uint32_t d, uint32_t a, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d), "r"(a), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
        "r"(r[30]), "r"(r[31]) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// N columns of this lane; the values are there after tc_wait_ld.
template <int N> __device__ __forceinline__ void tc_ld(uint32_t taddr, uint32_t* r) {
    if constexpr (N > 16) {
        tc_ld<16>(taddr, r);
        tc_ld<N - 16>(taddr + 16, r + 16);
    } else if constexpr (N == 16) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                       "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr) : "memory");
    } else if constexpr (N == 8) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
    } else {
        static_assert(N == 4, "columns of a load");
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
    }
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// K-major operand image, 128-byte swizzle, groups of eight rows 1024 bytes apart.
__device__ __forceinline__ uint64_t b_descriptor(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// binary16 x binary16 -> fp32, both K-major, 128 x N
__host__ __device__ constexpr uint32_t mma_idesc(int N) { return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24); }

// One lane of a converged warp, the same one every time.
__device__ __forceinline__ bool elect_lane() {
    uint32_t yes;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(yes));
    return yes != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void umma_cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t umma_cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ float ld_peer(uint32_t addr, uint32_t rank) {
    float v;
    uint32_t at;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
    return v;
}

__device__ __forceinline__ void arrive_peer(uint64_t* bar, uint32_t rank) {
    uint32_t at;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(bar)), "r"(rank));
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(at) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Barrier of the expanding warps; true when `ok` was true for all of them.
__device__ __forceinline__ bool expand_barrier(bool ok) {
    uint32_t all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbarrier.cta.red.and.pred p, 1, %2, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(all) : "r"((uint32_t)ok), "n"(kExpandThreads) : "memory");
    return all != 0;
}
__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void add_release_gpu(uint32_t* p, uint32_t v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// a += b, two floats at a time
__device__ __forceinline__ void add_pair(float2& a, uint32_t b0, uint32_t b1) {
    asm("{\n\t.reg .b64 x, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 z, {%0, %1};\n\tadd.rn.f32x2 z, z, x;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "+f"(a.x), "+f"(a.y) : "r"(b0), "r"(b1));
}

// Byte of (row n, column c of the matrix) in the operand images of 2 * NB rows.
template <int NB> __device__ __forceinline__ size_t image_at(int n, int c) {
    return (size_t)(c >> 6) * (NB * 256) + (size_t)(n * 128 + ((((c >> 3) & 7) ^ (n & 7)) << 4) + (c & 7) * 2);
}
// The mark of an input that binary16 cannot hold: +0 above, -0 below, which no other input gives (what rounds to +0 is not
// negative, and -0 leaves a remainder of +0).
constexpr uint32_t kBadLo = 0x8000u;
__device__ __forceinline__ bool too_large(float x) { return !(fabsf(x) < 65520.f); }
__device__ __forceinline__ uint32_t split_pair(float a, float b, uint32_t& lo, bool& large) {
    const bool la = too_large(a), lb = too_large(b);
    if (la) a = 0.f;
    if (lb) b = 0.f;
    large = large || la || lb;
    const __half h0 = __float2half_rn(a), h1 = __float2half_rn(b);
    const __half l0 = __float2half_rn(a - __half2float(h0)), l1 = __float2half_rn(b - __half2float(h1));
    lo = (uint32_t)__half_as_ushort(l0) | ((uint32_t)__half_as_ushort(l1) << 16) | (la ? kBadLo : 0u) | (lb ? kBadLo << 16 : 0u);
    return (uint32_t)__half_as_ushort(h0) | ((uint32_t)__half_as_ushort(h1) << 16);
}
// These write inputs into the images; true where one of them is marked.
template <int NB> __device__ __forceinline__ bool put_value(uint8_t* images, int b, int c, float x) {
    const bool large = too_large(x);
    if (large) x = 0.f;
    const __half hi = __float2half_rn(x), lo = __float2half_rn(x - __half2float(hi));
    uint8_t* at = images + image_at<NB>(b, c);
    *reinterpret_cast<__half*>(at) = hi;
    *reinterpret_cast<__half*>(at + NB * 128) = large ? __ushort_as_half((unsigned short)kBadLo) : lo;
    return large;
}
template <int NB> __device__ __forceinline__ bool put_split(uint8_t* images, int b, int c, const float (&x)[8]) {
    bool large = false;
    uint4 hi, lo;
    hi.x = split_pair(x[0], x[1], lo.x, large); hi.y = split_pair(x[2], x[3], lo.y, large);
    hi.z = split_pair(x[4], x[5], lo.z, large); hi.w = split_pair(x[6], x[7], lo.w, large);
    uint8_t* at = images + image_at<NB>(b, c);
    *reinterpret_cast<uint4*>(at) = hi;
    *reinterpret_cast<uint4*>(at + NB * 128) = lo;
    return large;
}
// Columns c .. c + 7 (those below n) of batch column b; src points at column c.
template <int NB> __device__ __forceinline__ bool put_eight(uint8_t* images, int b, int c, int n, const float* src, bool vec) {
    if (c + 8 <= n) {
        float x[8];
        if (vec) {
            const float4 u = __ldg(reinterpret_cast<const float4*>(src)), v = __ldg(reinterpret_cast<const float4*>(src) + 1);
            x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = src[i];
        }
        return put_split<NB>(images, b, c, x);
    }
    bool large = false;
    for (int i = 0; c + i < n; ++i) large |= put_value<NB>(images, b, c + i, src[i]);
    return large;
}

// Sets those sums to NaN, where they lie, that have a marked input in a column that their row keeps: out[b * ld] for the batch
// columns b.  Marks are rare, so the images and the items' headers are simply read again: first which columns of each window and
// batch column are marked, into shared memory that is free at the time (scratch), then each header once.  WARPS: the
// expanding warps of a product together, or the one that copies a time loop's inputs (the former cost two 2048-unit
// LSTM layers 2 % without any marks).  buffer: which of a time loop's buffers of images, whose sums lie [batch column][row
// of the group]; -1: a product's.
template <int NB, int MT, int WARPS>
__device__ __noinline__ void spoil_sums(const UmmaArgs& a, int p_idx, int cta, int warp, int buffer, uint8_t* scratch, int scratch_bytes, float* out, long long ld) {
    constexpr int kPer = 4 / MT;                           // windows of a round
    const UmmaPart& pt = a.part[p_idx];
    const UmmaCta me = pt.ctas[cta];
    const int lane = threadIdx.x & 31, nw = me.nw, seg_words = pt.seg_words, segs = 32 / seg_words, chunk = scratch_bytes / (NB * 8);
    const uint8_t *stream = pt.stream + (size_t)me.off128 * 128, *images = pt.xp + ((size_t)max(buffer, 0) * pt.windows + me.w0) * (NB * 256);
    const uint2* rounds = reinterpret_cast<const uint2*>(pt.rounds) + me.table;
    uint32_t seg_off[4 * MT];                              // the lane's row segment in each quadrant: where its headers start in an item
    int to[4 * MT];                                        // and its row in `out`
#pragma unroll
    for (int i = 0; i < 4 * MT; ++i) {
        const UmmaQuad q = pt.quads[(size_t)me.group * MT * 4 + i];
        seg_off[i] = lane < q.nrows ? (uint32_t)((q.row0 + lane) / pt.block_r - q.row0 / pt.block_r) * (uint32_t)(segs * 16) : 0u;
        to[i] = (buffer < 0 ? q.out0 : i * 32) + lane;
    }
    auto sync = [] { if (WARPS > 1) expand_barrier(true); else __syncwarp(); };
    for (int c0 = 0; c0 < nw; c0 += chunk) {
        const int n = min(chunk, nw - c0);
        sync();
#pragma unroll 4
        for (int i = warp * 32 + lane; i < n * a.nb * 8; i += WARPS * 32) {        // eight columns of a batch column
            const int w = (i >> 3) / a.nb, b = (i >> 3) - w * a.nb;
            const uint8_t* at = images + (size_t)(c0 + w) * (NB * 256) + b * 128 + (i & 7) * 16;
            const uint4 h = __ldcg(reinterpret_cast<const uint4*>(at)), l = __ldcg(reinterpret_cast<const uint4*>(at + NB * 128));
            auto pair = [](uint32_t hi, uint32_t lo) {
                return (uint32_t)((hi & 0xffffu) == 0u && (lo & 0xffffu) == kBadLo) | (uint32_t)(hi >> 16 == 0u && lo >> 16 == kBadLo) << 1;
            };
            scratch[(w * NB + b) * 8 + ((i & 7) ^ (b & 7))] = (uint8_t)(pair(h.x, l.x) | pair(h.y, l.y) << 2 | pair(h.z, l.z) << 4 | pair(h.w, l.w) << 6);
        }
        sync();
#pragma unroll 2
        for (int i = warp; i < n * MT; i += WARPS) {
            const int w = i / MT, mt = i - w * MT, rd = (c0 + w) / kPer, nj = min(4, nw * MT - 4 * rd), len = umma_unit_len(MT, a.flush, nj);
            int j = 0;
            while (j < 3 && (umma_place(MT, len, j).mt != mt || umma_place(MT, len, j).window != (c0 + w) % kPer)) ++j;
            const uint8_t* round = stream + (size_t)__ldg(rounds + rd).x * 16;
            const uint4 items = __ldg(reinterpret_cast<const uint4*>(round) + j);
            const uint32_t item[4] = {items.x, items.y, items.z, items.w};
#pragma unroll 1
            for (int s = 0; s < segs; ++s) {
                uint4 h[4];                                // (all four loaded in front of the stores)
#pragma unroll
                for (int quad = 0; quad < 4; ++quad) h[quad] = __ldg(reinterpret_cast<const uint4*>(round + item[quad] + seg_off[MT == 2 ? mt * 4 + quad : quad]) + s);
#pragma unroll 2
                for (int b = 0; b < a.nb; ++b) {
                    const uint32_t m = smem_u32(scratch) + (uint32_t)((w * NB + b) * 8), m0 = lds32(m), m1 = lds32(m + 4);
                    if ((m0 | m1) == 0u) continue;
#pragma unroll
                    for (int quad = 0; quad < 4; ++quad) {
                        const uint32_t hit = segs == 1 ? (m0 & h[quad].z) | (m1 & h[quad].w) : segs == 2 ? (s ? m1 : m0) & h[quad].z : ((s < 2 ? m0 : m1) >> (16 * (s & 1))) & h[quad].z;
                        if (((h[quad].x >> lane) & 1u) && hit) out[to[MT == 2 ? mt * 4 + quad : quad] + b * ld] = __int_as_float(0x7fffffff);
                    }
                }
            }
        }
    }
}

// One column segment of W words: the lane's row of it, zeros where the row is not kept.
template <int W>
__device__ __forceinline__ void expand_segment(uint32_t item, uint32_t header, int lane, uint32_t* r) {
    const uint4 h = lds128(header);
    const uint32_t kept = (h.x >> lane) & 1u, step = (uint32_t)__popc(h.x) * 16u;
    uint32_t p = item + h.y + (uint32_t)__popc(h.x & ((1u << lane) - 1u)) * 16u;
#pragma unroll
    for (int j = 0; j < W; j += 4, p += step)
        asm volatile(
            "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
            "@q ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
            : "=&r"(r[j]), "=&r"(r[j + 1]), "=&r"(r[j + 2]), "=&r"(r[j + 3]) : "r"(p), "r"(kept));
}

// Shared memory: the two rings (a bare product reuses them for the CTA's sums when the loop is over), then the time loop's
// sums and cell states, then barriers.
struct UmmaSmem {
    uint32_t w, part, cs, bars, total;         // (the inputs start at 0)
    __host__ __device__ UmmaSmem(int mode, int NB, int MT, int x_depth, int w_bytes) {
        const uint32_t sums = (uint32_t)(NB * MT * 512);
        w = (uint32_t)(x_depth * x_windows(NB, MT) * NB * 256);
        const uint32_t end = w + (uint32_t)w_bytes;
        part = mode ? end : 0u;
        cs = part + sums;
        bars = mode ? cs + sums / 4u : end > sums ? end : sums;
        total = bars + 512u + 1024u;
    }
};

template <int NB, int MT, int MODE>
__global__ void __launch_bounds__(kUmmaThreads, 1) csb_umma_kernel(const __grid_constant__ UmmaArgs a) {
    constexpr int N = 2 * NB;                             // hi and lo rows of the operand
    constexpr int kWin = N * 128;                         // bytes of a window's image
    constexpr int XW = x_windows(NB, MT), kXStage = XW * kWin;
    // lo rows with an instruction and sums of their own, which stay in TMEM until the end; else the two kinds side by side.  Twice the
    // instructions for half the loads from TMEM (those of 64 columns took 17 of 44 us): 8192 x 8192 at 4x, batch 64, 44.4 ->
    // 29.6 us, two 2048-unit LSTM layers with 32 sequences 23.8 -> 20.9 us a step; batch 8 19.1 -> 19.8.
    constexpr bool kSplit = NB >= 32;
    constexpr int DW = kSplit ? NB : N;                   // columns of a unit's sums
    constexpr int kLoCol = 128;                           // where the lo rows' own begin
    constexpr int DB = (kSplit ? kLoCol : kDCols) / DW;   // buffers of sums, one per unit (a power of two)
    constexpr int CN = NB * MT / 4;                       // batch columns whose sums a warp keeps
    constexpr int kRows = 128 * MT;
    static_assert((!kSplit || kLoCol + MT * NB <= kDCols) && kDCols + kASlots * 32 <= 512 && DB >= 2, "TMEM");
    const int XD = a.x_depth;
    const UmmaSmem L(MODE, NB, MT, XD, a.w_bytes);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars);
    uint64_t *xfull = bars, *xempty = xfull + kMaxXDepth, *wfull = xempty + kMaxXDepth, *wempty = wfull + kWRounds;
    uint64_t *afull = wempty + kWRounds, *aempty = afull + 2, *dfull = aempty + 2, *dempty = dfull + DB, *pfull = dempty + DB, *xdone = pfull + 1;
    uint64_t *sums = xdone + 1, *spoilt = sums + 1;
    volatile uint32_t* s_dead = reinterpret_cast<volatile uint32_t*>(spoilt + 1);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(spoilt + 1) + 1;
    volatile uint32_t* w_at = reinterpret_cast<volatile uint32_t*>(spoilt + 2);       // where a round of values lies in its ring
    // Are there marks in the CTA's windows?  Time loop: the call and tick of the latest mark in the images (a copy, 16 bytes); then
    // whether a state of the CTA's own is marked; then the number of ticks whose sums have been gone through.
    volatile uint32_t* s_bad = reinterpret_cast<volatile uint32_t*>(smem + L.bars + 384);
    static_assert((2 * kMaxXDepth + 2 * kWRounds + 4 + 2 * DB + 5) * 8 + kWRounds * 4 <= 384, "the barriers end before");
    float* part = reinterpret_cast<float*>(smem + L.part);        // the CTA's sums: [batch column][row of the group]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (MODE == 0) pdl_launch_dependents();               // (a time loop may run for long: nothing need wait on its SMs so long)
    int p_idx = 0, cta0 = 0;                              // which product (layer) this CTA works for, and its first CTA
    while (p_idx + 1 < a.n_parts && (int)blockIdx.x >= a.part[p_idx].cta_end) { cta0 = a.part[p_idx].cta_end; ++p_idx; }
    const UmmaPart& pt = a.part[p_idx];
    const UmmaCta* me = pt.ctas + ((int)blockIdx.x - cta0);
    const int nw = me->nw, w0 = me->w0, F = a.flush, T_ = MODE ? a.T : 1;
    const int ntw = nw * MT, rounds = (ntw + 3) / 4;
    if (threadIdx.x == 0) {
        for (int i = 0; i < XD; ++i) { mbar_init(xfull + i, 1); mbar_init(xempty + i, 1); }
        for (int i = 0; i < kWRounds; ++i) { mbar_init(wfull + i, 1); mbar_init(wempty + i, kUmmaExpandWarps); }
        for (int i = 0; i < 2; ++i) { mbar_init(afull + i, kUmmaExpandWarps); mbar_init(aempty + i, 1); }
        for (int i = 0; i < DB; ++i) { mbar_init(dfull + i, 1); mbar_init(dempty + i, kUmmaExpandWarps / MT); }
        mbar_init(pfull, (uint32_t)a.S);
        mbar_init(xdone, 1);
        mbar_init(sums, kUmmaExpandWarps);
        mbar_init(spoilt, 1);
        *s_dead = 0u;
        s_bad[0] = s_bad[1] = s_bad[4] = s_bad[5] = 0u;
        mbar_fence_init();
    }
    if (warp == kUmmaExpandWarps) tc_alloc(smem_u32(s_tmem), 512);
    tc_fence_before();
    __syncthreads();
    if (MODE && a.S > 1) umma_cluster_barrier();          // the peers' barriers are there before anybody arrives on them
    tc_fence_after();
    // (all of TMEM is this CTA's, so it starts at column 0: as a constant the addresses stay in uniform registers)
    constexpr uint32_t tmem = 0u, a_base = kDCols;
    if (threadIdx.x == 0 && *s_tmem != 0u) { *s_dead = 1u; *(volatile uint32_t*)a.status = (uint32_t)kDevCopyTimeout; }

    // A wait gives up after a second, or as soon as another one of the CTA has given up.  What a product's wait stands behind
    // must be this kernel's own work: each role passes pdl_wait before its first wait that needs the inputs, so that the
    // time of the work in front does not count.
    auto gave_up = [&](unsigned int& spins, unsigned long long& t0, unsigned long long limit, uint32_t code) -> bool {
        if ((++spins & 255u) != 0) return false;
        if (*s_dead) return true;
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > limit) { *s_dead = 1u; *(volatile uint32_t*)a.status = code; return true; }
        return false;
    };
    // (in the time loop a wait may last as long as the one for other CTAs)
    const unsigned long long limit = MODE ? kCopyWaitNs + a.limit_ns : kCopyWaitNs;
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        if (mbar_try_wait(bar, parity)) return true;
        unsigned long long t0 = 0;
        unsigned int spins = 0;
        while (!mbar_try_wait_parked(bar, parity, 4000u)) if (gave_up(spins, t0, limit, kDevCopyTimeout)) return false;
        return true;
    };
    // Time loop: every CTA with a step in an earlier tick than this layer's step t has finished it.
    auto wait_tick = [&](int t, uint32_t never) -> bool {
        uint32_t need = never;
        for (int l = 0; l < a.n_parts; ++l)
            need += (uint32_t)(a.part[l].cta_end - (l ? a.part[l - 1].cta_end : 0)) * (uint32_t)min(max(t + p_idx - l, 0), T_);
        unsigned long long t0 = 0;
        unsigned int spins = 0;
        while ((int32_t)(ld_acquire_gpu(a.count) - need) < 0) if (gave_up(spins, t0, a.limit_ns, kDevBarrierTimeout)) return false;
        return true;
    };
    // Time loop: there is a marked input in what the part reads in that tick.
    auto mark = [&](const UmmaPart& part_of, int tick) {
        *reinterpret_cast<uint2*>(part_of.bad + 4 * (tick & 1)) = make_uint2(a.call, (uint32_t)tick + 1u);
    };
    float2 acc[CN / 2];
#pragma unroll
    for (int i = 0; i < CN / 2; ++i) acc[i] = make_float2(0.f, 0.f);
    const int quad = warp & 3, slot = warp >> 2;          // expanding warps: lanes of the tile, which tile-window of a round
    const int my_mt = MT == 2 ? slot >> 1 : 0, my_b0 = MT == 2 ? (slot & 1) * CN : slot * CN;      // and whose sums the warp keeps
    const UmmaQuad* quads = pt.quads + (size_t)me->group * MT * 4;
    if (warp < kUmmaExpandWarps) {
        const int seg_words = pt.seg_words, segs = 32 / seg_words;
        uint32_t seg_off[MT];                             // the lane's row segment: where its headers start in an item
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            const UmmaQuad q = quads[mt * 4 + quad];
            seg_off[mt] = lane < q.nrows ? (uint32_t)((q.row0 + lane) / pt.block_r - q.row0 / pt.block_r) * (uint32_t)(segs * 16) : 0u;
        }
        const uint32_t rank = a.S > 1 ? umma_cluster_rank() : 0u;
        float* cs = reinterpret_cast<float*>(smem + L.cs);
        // the time loop's share of this warp: (tile of 32 units, batch column) pairs
        const int tasks = MODE ? (MT * a.nb - (int)rank + a.S - 1) / a.S : 0;
        if (MODE)
            for (int j = warp; j < tasks; j += kUmmaExpandWarps) {
                const int k = (int)rank + a.S * j, ut = k / a.nb, b = k - ut * a.nb;
                const UmmaQuad q = quads[ut * 4];
                cs[j * 32 + lane] = lane < q.nrows ? __ldg(a.state0 + ((size_t)p_idx * a.nb + b) * a.H + q.row0 + lane) : 0.f;
            }
        bool ok = true;
        // The warp's share of sums in TMEM from this column on, added to its own; both: hi rows' and, NB columns on, lo rows'.
        auto take = [&](uint32_t column, bool both) {
            constexpr int CP = CN < 16 ? CN : 16;         // columns at a time: what the registers hold beside the sums
            const uint32_t d = tmem + ((uint32_t)quad << 21) + column + (uint32_t)my_b0;
#pragma unroll
            for (int c = 0; c < CN; c += CP) {
                uint32_t v[CP], lo[CP];
                tc_ld<CP>(d + c, v);
                if (both) tc_ld<CP>(d + NB + c, lo);
                tc_wait_ld();
#pragma unroll
                for (int i = 0; i < CP / 2; ++i) {
                    if (both) {
                        float2 h = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                        add_pair(h, lo[2 * i], lo[2 * i + 1]);
                        add_pair(acc[c / 2 + i], __float_as_uint(h.x), __float_as_uint(h.y));
                    } else add_pair(acc[c / 2 + i], v[2 * i], v[2 * i + 1]);
                }
            }
        };
        // Sums of a unit (by the running number).
        auto drain = [&](uint32_t run) {
            const uint32_t buf = run % DB;
            ok = __all_sync(0xffffffffu, wait(dfull + buf, (run / DB) & 1u));
            if (!ok) return;
            tc_fence_after();
            take(buf * DW, !kSplit);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(dempty + buf);
        };
        uint32_t ws = 0, w_par = 0, half = 0, a_par = 1, run = 0;     // slot and parity of the values and of the operand; running number of units
        for (int t = 0; t < T_ && ok; ++t) {
            int before = 0;                               // units of the round in front, whose sums are still in TMEM
            for (int rd = 0; rd < rounds && ok; ++rd) {
                const int nj = min(4, ntw - 4 * rd), len = umma_unit_len(MT, F, nj);
                ok = __all_sync(0xffffffffu, wait(wfull + ws, w_par));
                if (!ok) break;
                uint32_t r[32];
                if (slot < nj) {
                    const uint32_t blob = smem_u32(smem) + L.w + w_at[ws], item = blob + lds32(blob + 4u * warp);
                    const uint32_t header = item + (umma_place(MT, len, slot).mt ? seg_off[MT - 1] : seg_off[0]);
                    if (seg_words == 32) expand_segment<32>(item, header, lane, r);
                    else if (seg_words == 16) { expand_segment<16>(item, header, lane, r); expand_segment<16>(item, header + 16, lane, r + 16); }
                    else
#pragma unroll
                        for (int s = 0; s < 4; ++s) expand_segment<8>(item, header + 16 * s, lane, r + 8 * s);
                }
                ok = __all_sync(0xffffffffu, wait(aempty + half, a_par));      // (fresh: ends at once)
                if (!ok) break;
                tc_fence_after();
                if (slot < nj) tc_st32(a_base + ((uint32_t)quad << 21) + (half * 4u + (uint32_t)slot) * 32u, r);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { mbar_arrive(afull + half); mbar_arrive(wempty + ws); }
                if (++ws == kWRounds) { ws = 0; w_par ^= 1u; }
                half ^= 1u;
                a_par ^= half ^ 1u;
                if (MODE == 0 && rd == 1) pdl_wait();     // (two rounds of operands fit in TMEM without the inputs)
                // The sums of the round in front, while this one's products run.  (Half of the warps before they expand and half
                // after it: a quarter slower.)
                for (int u = my_mt; u < before && ok; u += MT) drain(run + u);
                run += (uint32_t)before;
                before = (nj + (MT == 2 ? 0 : len - 1)) >> (len - 1);       // nj / len, rounded up for one tile; len is 1 or 2
            }
            if (MODE == 0 && rounds == 1) pdl_wait();
            for (int u = my_mt; u < before && ok; u += MT) drain(run + u);
            run += (uint32_t)before;
            if (kSplit && ok) { take(kLoCol + (uint32_t)(my_mt * NB), false); tc_fence_before(); }   // the lo rows' sums, complete with the tile's last unit
            if constexpr (MODE != 0) {
            // ---- the step's sums are complete: cluster, gates, h_t
#pragma unroll
            for (int i = 0; i < CN / 2; ++i) {
                float* at = part + (my_b0 + 2 * i) * kRows + my_mt * 128 + quad * 32 + lane;
                at[0] = acc[i].x; at[kRows] = acc[i].y;
                acc[i] = make_float2(0.f, 0.f);
            }
            if (ok && s_bad[0] == a.call && s_bad[1] == (uint32_t)(t + p_idx + 1)) {
                const uint32_t par = s_bad[5] & 1u;       // the copying warp goes through them
                __syncwarp();
                if (lane == 0) mbar_arrive(sums);
                ok = __all_sync(0xffffffffu, wait(spoilt, par));
            }
            ok = expand_barrier(ok);
            if (!ok) break;
            if (a.S > 1 && (int)threadIdx.x < a.S) arrive_peer(pfull, threadIdx.x);
            const bool more = t + 1 < T_;
            const int next = (t + p_idx + 1) & 1;         // the buffer of images that the next tick reads
            if (a.S > 1) {
                unsigned long long t0 = 0;
                unsigned int spins = 0;
                while (!mbar_try_wait_cluster(pfull, (uint32_t)t & 1u)) if (gave_up(spins, t0, limit, kDevBarrierTimeout)) { ok = false; break; }
                ok = __all_sync(0xffffffffu, ok);
            }
            // two of the warp's tasks at a time, so that their loads are in flight together (one after the other 4 us a step)
            for (int j0 = warp; j0 < tasks && ok; j0 += 2 * kUmmaExpandWarps) {
                float z[2][4], zb[2][4];
                uint32_t at[2];
                int u[2], b[2];
                bool live[2];
                const float* bl = a.bias[p_idx];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int j = min(j0 + p * kUmmaExpandWarps, tasks - 1), k = (int)rank + a.S * j, ut = k / a.nb;
                    b[p] = k - ut * a.nb;
                    const UmmaQuad q = quads[ut * 4];
                    u[p] = q.row0 + lane;
                    live[p] = lane < q.nrows && j0 + p * kUmmaExpandWarps < tasks;
                    at[p] = smem_u32(part) + (uint32_t)(b[p] * kRows + ut * 128 + lane) * 4u;
#pragma unroll
                    for (int gt = 0; gt < 4; ++gt) zb[p][gt] = bl && live[p] ? __ldg(bl + (size_t)gt * a.H + u[p]) : 0.f;
                }
                auto range = [&](int s, float (&v)[2][4]) {
#pragma unroll
                    for (int p = 0; p < 2; ++p)
#pragma unroll
                        for (int gt = 0; gt < 4; ++gt) v[p][gt] = a.S > 1 ? ld_peer(at[p] + gt * 128u, (uint32_t)s) : __uint_as_float(lds32(at[p] + gt * 128u));
                };
                range(0, z);
                for (int s = 1; s < a.S; ++s) {
                    float v[2][4];
                    range(s, v);
#pragma unroll
                    for (int p = 0; p < 2; ++p)
#pragma unroll
                        for (int gt = 0; gt < 4; ++gt) z[p][gt] += v[p][gt];
                }
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    if (!live[p]) continue;
                    if (bl) {
#pragma unroll
                        for (int gt = 0; gt < 4; ++gt) z[p][gt] += zb[p][gt];
                    }
                    float* state = cs + (j0 + p * kUmmaExpandWarps) * 32 + lane;
                    float st = *state, h;
                    if (MODE == 1) h = lstm_cell(z[p][0], z[p][1], z[p][2], z[p][3], st);
                    else st = h = gru_cell(z[p][0], z[p][1], z[p][2], z[p][3], st);
                    *state = st;
                    if (too_large(h)) s_bad[4] = 1u;
                    if (more) put_value<NB>(pt.xp + (size_t)next * pt.windows * kWin, b[p], a.in_size[p_idx] + u[p], h);
                    if (p_idx + 1 < a.n_parts) {
                        const UmmaPart& above = a.part[p_idx + 1];
                        put_value<NB>(above.xp + (size_t)next * above.windows * kWin, b[p], u[p], h);
                    } else if (a.y) a.y[((size_t)t * a.nb + b[p]) * a.H + u[p]] = h;
                    if (!more) {
                        const size_t e = ((size_t)p_idx * a.nb + b[p]) * a.H + u[p];
                        if (a.hT) a.hT[e] = h;
                        if (MODE == 1 && a.cT) a.cT[e] = st;
                    }
                }
            }
            // (in front of the barrier: a warp that gives up takes the others along, which would wait for it at the next one)
            if (warp == 0 && p_idx == 0 && more && ok) ok = __all_sync(0xffffffffu, wait(xdone, (uint32_t)t & 1u));
            ok = expand_barrier(ok);
            if (!ok) break;
            if (threadIdx.x == 0) {
                if (s_bad[4]) {
                    s_bad[4] = 0u;
                    mark(pt, t + p_idx + 1);
                    if (p_idx + 1 < a.n_parts) mark(a.part[p_idx + 1], t + p_idx + 1);
                }
                __threadfence();
                add_release_gpu(a.count, 1u);
            }
            }
        }
    } else if (warp == kUmmaExpandWarps) {
        // The whole warp runs along, so that addresses and descriptors live in uniform registers, and one lane issues (with a
        // single lane running, a tile-window took this warp 1100 cycles: it was what the others waited for).
        const bool leader = elect_lane();
        if (MODE == 0) pdl_wait();
        bool ok = true;
        uint32_t half = 0, a_par = 0, xs = 0, x_par = 0, buf = 0, d_par = 1;
        const uint64_t x_desc = b_descriptor(smem_u32(smem));
        for (int t = 0; t < T_ && ok; ++t)
            for (int rd = 0; rd < rounds && ok; ++rd) {
                const int nj = min(4, ntw - 4 * rd), len = umma_unit_len(MT, F, nj);
                ok = __all_sync(0xffffffffu, wait(afull + half, a_par) && wait(xfull + xs, x_par));
                uint64_t x = x_desc + (uint64_t)((xs * kXStage) >> 4);
                for (int j0 = 0; j0 < nj && ok; j0 += len) {
                    if (XW < 4 / MT && j0 == XW) {        // the second stage of the round
                        if (leader) tc_commit(xempty + xs);
                        if (++xs == (uint32_t)XD) { xs = 0; x_par ^= 1u; }
                        ok = wait(xfull + xs, x_par);
                        x = x_desc + (uint64_t)((xs * kXStage) >> 4);
                    }
                    ok = __all_sync(0xffffffffu, ok && wait(dempty + buf, d_par));
                    if (!ok) break;
                    tc_fence_after();
                    if (leader) {
#pragma unroll 2
                        for (int j = j0; j < min(j0 + len, nj); ++j) {
                            const UmmaPlace at = umma_place(MT, len, j);
                            const uint64_t b = x + (uint64_t)((at.window % XW * kWin) >> 4);
                            const uint32_t lo = tmem + kLoCol + at.mt * NB;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t op = a_base + (half * 4u + (uint32_t)j) * 32u + k * 8;
                                tc_mma_f16(tmem + buf * DW, op, b + (uint64_t)(2 * k), mma_idesc(DW), j != j0 || k != 0);
                                if (kSplit) tc_mma_f16(lo, op, b + (uint64_t)(NB * 8 + 2 * k), mma_idesc(NB), rd != 0 || at.window != 0 || k != 0);
                            }
                        }
                        tc_commit(dfull + buf);
                    }
                    __syncwarp();
                    if (++buf == DB) { buf = 0; d_par ^= 1u; }
                }
                if (!ok) break;
                if (leader) { tc_commit(aempty + half); tc_commit(xempty + xs); }
                __syncwarp();
                if (++xs == (uint32_t)XD) { xs = 0; x_par ^= 1u; }
                half ^= 1u;
                a_par ^= half ^ 1u;
            }
    } else if (warp == kUmmaExpandWarps + 1) {
        if (!MODE) pdl_wait();                            // the packed inputs belong to the work in front on the stream
        bool ok = true;
        uint32_t at = 0, par = 1;
        for (int t = 0; t < T_; ++t) {
            bool marked = false;
            if (lane == 0) {
                const uint8_t* src = pt.xp + (size_t)w0 * kWin;
                const uint32_t* marks = pt.bad + 4 * ((t + p_idx) & 1);
                if (MODE) {
                    src += (size_t)((t + p_idx) & 1) * pt.windows * kWin;
                    ok = wait_tick(t, a.never);
                    fence_proxy_async_all();              // what others have stored is read by copies
                }
                for (int w = 0; w < nw && ok; w += XW) {
                    ok = wait(xempty + at, par);
                    if (!ok) break;
                    const uint32_t bytes = (uint32_t)min(XW, nw - w) * kWin;
                    if (MODE && w == 0) {                 // (with the tick's first images: the tick in front has been read)
                        mbar_expect_tx(xfull + at, bytes + 16u);
                        bulk_g2s(const_cast<uint32_t*>(s_bad), marks, 16u, xfull + at);
                    } else mbar_expect_tx(xfull + at, bytes);
                    bulk_g2s(smem + at * kXStage, src + (size_t)w * kWin, bytes, xfull + at);
                    if (++at == (uint32_t)XD) { at = 0; par ^= 1u; }
                }
                if (MODE && ok) marked = __ldcg(marks) == a.call && __ldcg(marks + 1) == (uint32_t)(t + p_idx + 1);
            }
            if (MODE) {
                if (!__shfl_sync(0xffffffffu, ok, 0)) break;
                if (!__shfl_sync(0xffffffffu, marked, 0)) continue;
                if (!__all_sync(0xffffffffu, wait(sums, s_bad[5] & 1u))) break;
                // (the inputs' ring is free: this warp fills it, and every product of the step is done)
                spoil_sums<NB, MT, 1>(a, p_idx, (int)blockIdx.x - cta0, 0, (t + p_idx) & 1, smem, (int)L.w, part, kRows);
                fence_proxy_async_all();                  // (the next tick's copies go over the scratch)
                __syncwarp();
                if (lane == 0) { s_bad[5] = s_bad[5] + 1u; mbar_arrive(spoilt); }
                __syncwarp();
            }
        }
    } else if (warp == kUmmaExpandWarps + 2) {
        if (lane == 0) {                                  // (written at plan time: the copies need not wait for the work in front)
            const uint8_t* src = pt.stream + (size_t)me->off128 * 128;
            const uint2* table = reinterpret_cast<const uint2*>(pt.rounds) + me->table;
            // Rounds lie one behind the other in the ring, each in one piece; the next one goes where the oldest have left room.
            const uint32_t cap = (uint32_t)a.w_bytes;
            bool ok = true;
            uint32_t head = 0, tail = 0, there = 0, at = 0, old = 0, old_par = 0;      // there: rounds in the ring, from slot `old` on
            int freed = 0;                                // (the expanding warps are done with two rounds before they need the inputs)
            uint2 next = __ldg(table);
            for (int t = 0; t < T_ && ok; ++t)
                for (int rd = 0; rd < rounds && ok; ++rd) {
                    const uint2 now = next;
                    next = __ldg(table + (rd + 1 < rounds ? rd + 1 : 0));
                    for (;;) {
                        if (there == 0) { head = tail = 0; break; }
                        if (there < kWRounds) {
                            if (head > tail) {
                                if (cap - head >= now.y) break;
                                if (tail > now.y) { head = 0; break; }
                            } else if (tail > head && tail - head > now.y) break;
                        }
                        if (MODE == 0 && freed++ == 2) pdl_wait();
                        ok = wait(wempty + old, old_par);
                        if (!ok) break;
                        if (++old == kWRounds) { old = 0; old_par ^= 1u; }
                        --there;
                        tail = w_at[old];
                    }
                    if (!ok) break;
                    w_at[at] = head;
                    mbar_expect_tx(wfull + at, now.y);
                    bulk_g2s(smem + L.w + head, src + (size_t)now.x * 16, now.y, wfull + at);
                    head += now.y;
                    ++there;
                    if (++at == kWRounds) at = 0;
                }
        }
    } else if (MODE == 0) {                               // (as a block of its own behind these roles it cost 8192 x 8192 at batch 64 2.6 of 28 us)
        pdl_wait();
        const uint4* words = reinterpret_cast<const uint4*>(pt.bad) + w0 * (NB / 16);
        uint32_t any = 0;
#pragma unroll 4
        for (int i = lane; i < nw * (NB / 16); i += 32) {
            const uint4 u = __ldcg(words + i);
            any |= u.x | u.y | u.z | u.w;
        }
        if (any) s_bad[0] = 1u;
    } else if (p_idx == 0) {
        // x_{t+1}, shared between the CTAs of the first layer, while step t runs
        const int I = a.in_size[0], chunks = (I + 7) / 8;
        bool ok = true;
        for (int t = 0; t + 1 < T_ && ok; ++t) {
            ok = __all_sync(0xffffffffu, lane != 0 || wait_tick(t, t == a.never_step ? kNever : a.never));
            if (!ok) break;
            uint8_t* images = pt.xp + (size_t)((t + 1) & 1) * pt.windows * kWin;
            for (int i = (int)blockIdx.x * 32 + lane; i < chunks * a.nb; i += pt.cta_end * 32) {
                const int b = i / chunks, c = (i - b * chunks) * 8;
                if (put_eight<NB>(images, b, c, I, a.x + ((size_t)(t + 1) * a.nb + b) * I + c, a.x_vec != 0)) mark(pt, t + 1);
            }
            __syncwarp();
            if (lane == 0) { __threadfence(); mbar_arrive(xdone); }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool dead = *s_dead != 0u;
    if (dead) {
        // a wait gave up (the status word says so): copies and tensor instructions that may still be in flight get a bounded
        // time to end before the CTA's memories go away, and nothing is written
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    if (warp == kUmmaExpandWarps) tc_dealloc(tmem, 512);
    if (MODE) {
        if (a.S > 1) umma_cluster_barrier();              // nobody leaves before everybody has read
        return;
    }
    pdl_wait();                                           // Y belongs to the work in front
    const bool marked = s_bad[0] != 0u && !dead && warp < kUmmaExpandWarps;
    if (a.S == 1) {
        if (!dead && warp < kUmmaExpandWarps) {
            const UmmaQuad q = quads[my_mt * 4 + quad];
            if (lane < q.nrows)
#pragma unroll
                for (int i = 0; i < CN; ++i)
                    if (my_b0 + i < a.nb) pt.Y[(long long)(my_b0 + i) * a.ldy + q.out0 + lane] = i & 1 ? acc[i / 2].y : acc[i / 2].x;
        }
        if (marked) spoil_sums<NB, MT, kUmmaExpandWarps>(a, 0, (int)blockIdx.x, warp, -1, smem, (int)L.w, pt.Y, a.ldy);
        return;
    }
    if (warp < kUmmaExpandWarps)
#pragma unroll
        for (int i = 0; i < CN / 2; ++i) {
            float* at = part + (my_b0 + 2 * i) * kRows + my_mt * 128 + quad * 32 + lane;
            at[0] = acc[i].x; at[kRows] = acc[i].y;
        }
    __syncthreads();
    umma_cluster_barrier();
    // every CTA adds the ranges, in range order, for its share of the quadrants
    const uint32_t rank = umma_cluster_rank(), base = smem_u32(part);
    if (!dead && warp < kUmmaExpandWarps) {
        const int mine = (4 * MT - (int)rank + a.S - 1) / a.S;         // quadrants rank, rank + S, ..
        for (int i0 = warp; i0 < mine * a.nb; i0 += 2 * kUmmaExpandWarps) {
            float v[2][kUmmaMaxS];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int i = min(i0 + j * kUmmaExpandWarps, mine * a.nb - 1), qi = (int)rank + (i / a.nb) * a.S, b = i % a.nb;
                const uint32_t at = base + (uint32_t)(b * kRows + qi * 32 + lane) * 4u;
#pragma unroll
                for (int s = 0; s < kUmmaMaxS; ++s) v[j][s] = s < a.S ? ld_peer(at, (uint32_t)s) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int i = i0 + j * kUmmaExpandWarps, qi = (int)rank + (i / a.nb) * a.S, b = i % a.nb;
                if (i >= mine * a.nb) break;
                float sum = v[j][0];
#pragma unroll
                for (int s = 1; s < kUmmaMaxS; ++s) sum += v[j][s];
                const UmmaQuad q = quads[qi];
                if (lane < q.nrows) pt.Y[(long long)b * a.ldy + q.out0 + lane] = sum;
            }
        }
    }
    __syncthreads();
    umma_cluster_barrier();                               // nobody leaves before everybody has read
    if (marked) spoil_sums<NB, MT, kUmmaExpandWarps>(a, 0, (int)blockIdx.x, warp, -1, smem, (int)L.w, pt.Y, a.ldy);
}

}  // namespace csb
