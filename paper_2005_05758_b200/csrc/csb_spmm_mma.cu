// Tensor-core CSB-SpMM (batch >= 8, fp16 values, fp32 accumulation) for blocks whose width is not 16, 32 or a multiple of 64;
// those go through csb_umma_kernel.cuh, whose column segments need such widths (at 8 sizes from 512 x 512 to 8192 x 8192, 8 to
// 64 columns, 25x to 1000x, that kernel was the faster one at each, though its time does not fall with the kept weights, but for
// 8192 x 8192 at 1000x with 8 and 16 columns, 17.3 us here and 17.7 there).
//
// With a batch of vectors the product of a block's kernel matrix (m kept rows x n kept columns)
// with the gathered inputs (n x batch) of Section 4.3.1 is a small dense contraction, the one place
// on this path where tensor cores apply.  How it is laid out here:
//
//   * A warp works for one block-row over a range of block-columns and keeps that block-row's
//     outputs, all block_r rows x up to 64 batch columns, in the accumulator registers of
//     mma.sync.m16n8k16 for the whole range (several warps share a block-row's blocks; their sums
//     meet once, at the end).  The kernel matrix is the A operand with its kept rows put back at their
//     RowIdx positions: a lane finds the stored row behind an output row with a population count
//     on the block's 64-bit row mask and loads its fragment straight from the compact row-major
//     values (rows that are not kept give zero registers).  So nothing is scattered and nothing is
//     read-modify-written per block; the row indices never leave the registers.
//   * The inputs are packed once per call into binary16 pairs x = hi + lo (no input precision is
//     lost as long as |x| < 65504), one row of batch values per matrix column, and reach shared
//     memory as whole block-column tiles through a ring that all warps of the CTA share, so a tile
//     is fetched from L2 once per CTA and not once per block.  A tile spans up to four block-columns
//     (256 matrix columns), so that the warps hand tiles over a few times per CTA only.  The gather through ColIdx is done by
//     the operand load itself: every lane hands ldmatrix.trans the address of the tile row of one
//     kept column.  hi and lo are multiplied separately into the same accumulators.
//   * The weights of a warp come through its own ring of bulk copies, so warps with light and heavy
//     blocks do not wait for each other; they only meet at the input tiles, which a warp releases
//     in order whether it used them or not, the last warp to release a slot refilling it.
//   * A CTA covers RG block-rows x a range of block-columns (the planner's cut).  When a row group
//     is divided between S CTAs these are launched as one thread-block cluster and add their sums
//     through distributed shared memory, every CTA for a share of the rows and in the order of the
//     ranges, so results are bit-reproducible and no scratch in global memory is needed.
//   * More than 32 batch columns go through in tiles of 64 on 8 warps a CTA, or, where that plan does
//     not fit, in passes of 32; more than 64 in passes (the weights of the later ones come from L2).
#include <algorithm>
#include <cstdio>
#include <mutex>

#include "csb_host.hpp"
#include "csb_internal.hpp"
#include "csb_device.cuh"

namespace csb {

constexpr uint32_t kOffMaskM = 0x3fffffffu;
constexpr uint32_t kNoRow = 0xffffffffu;
constexpr size_t kSpmmStaticSmem = 256;       // the kernel's statically allocated shared memory (CTA descriptor, row table), rounded up

// One product of a launch: the layers of a recurrent stack that work on different steps at the same
// time share a launch, each with the CTAs of its own plan.
struct SpmmPart {
    const uint8_t* stream;
    const uint4* warp_desc;    // per warp: first chunk's offset, chunk count, sizes of its first three chunks
    const SpmmCta* ctas;
    const uint8_t* xp;         // packed inputs: one row of `pitch` bytes per matrix column
    float* Y;
    int rows, cols, RG, cta_end;   // cta_end: the part's CTAs end here in the grid
};
struct SpmmArgs {
    SpmmPart part[kMaxLayers];
    long long ldy;
    uint32_t* status;
    int n_parts, nb, block_r, block_c, tile_cols, S, x_depth, w_stages, pitch, tile_bytes;   // tile_cols: matrix columns per input tile
    int q_rows;                // rows of the largest row group the shared-memory carve-up must hold (RG * block_r of one product)
#ifdef CSB_SPMM_CLOCKS
    long long* clocks;         // instrumented build only: [CTA][warp][16] cycles per phase
#endif
};

#ifdef CSB_SPMM_CLOCKS
#define SPMM_LAP(i) do { const long long n_ = clock64(); sprof[i] += n_ - st_; st_ = n_; } while (0)
#else
#define SPMM_LAP(i) do { } while (0)
#endif

// Shared-memory carve-up, identical on host and device.  The small fixed part comes first; the two
// rings follow and are reused for the warps' partial sums once the main loop is over.
// Floats per row of a warp's sums in shared memory: the fragments go in with 8-byte stores and a row
// comes out with 16-byte loads, both without bank conflicts at this pitch.
__host__ __device__ constexpr int spmm_sum_pitch(int NT) { return NT == 1 ? 8 : 8 * NT + 8; }
__host__ __device__ constexpr size_t spmm_q_bytes(int NT, int group_rows) { return (size_t)8 * NT * (group_rows + 1) * 4; }

struct SpmmSmem {
    size_t wfull, xfull, wcnt, xcnt, dead, zero, rings, wring, xring, qsums, total;
    // q_bytes: room for the CTA's own sums of its row group
    __host__ __device__ SpmmSmem(int n_warps, int w_stages, int x_depth, int tile_bytes, int pitch, int MT, int NT, size_t q_bytes) {
        const int n_streams = n_warps;
        wfull = 0;
        xfull = wfull + (size_t)n_streams * w_stages * 8;
        wcnt = xfull + (size_t)x_depth * 8;
        xcnt = wcnt + (size_t)n_streams * w_stages * 4;
        dead = xcnt + (size_t)x_depth * 4;
        zero = (dead + 4 + 127) & ~(size_t)127;
        rings = (zero + (size_t)pitch + 127) & ~(size_t)127;
        wring = rings;
        xring = wring + (size_t)n_streams * w_stages * kSpmmStageBytes;
        const size_t ring_end = xring + (size_t)x_depth * tile_bytes;
        qsums = (rings + (size_t)n_warps * MT * 16 * spmm_sum_pitch(NT) * 4 + 127) & ~(size_t)127;
        const size_t sums_end = qsums + q_bytes;
        total = ring_end > sums_end ? ring_end : sums_end;
    }
};

// Pack X: fp32 [batch][cols] -> per column one row of binary16 values: the hi parts of the 8 * NT batch
// columns, then the lo parts (x = hi + lo); batch columns past nb are zero.
__global__ void csb_pack_x_kernel(const float* __restrict__ X, long long ldx, int nb, int cols, uint8_t* __restrict__ xp, int pitch, int NT) {
    pdl_launch_dependents();
    pdl_wait();                                    // X may come from the kernel in front; xp may still be read by it
    __shared__ float tile[64][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c0 = blockIdx.x * 32;
    const int cap = 8 * NT;
    for (int b = ty; b < cap; b += 8) tile[b][tx] = (b < nb && c0 + tx < cols) ? X[(long long)b * ldx + c0 + tx] : 0.f;
    __syncthreads();
    for (int idx = threadIdx.x; idx < 32 * cap; idx += blockDim.x) {
        const int c = idx / cap, b = idx % cap;
        if (c0 + c >= cols) break;
        const float x = tile[b][c];
        const __half hi = __float2half_rn(x);
        const __half lo = __float2half_rn(x - __half2float(hi));
        __half* row = reinterpret_cast<__half*>(xp + (size_t)(c0 + c) * pitch);
        row[b] = hi;
        row[cap + b] = lo;
    }
}

__device__ __forceinline__ void mma_m16n8k16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ uint32_t atom_add_acq_rel_shared(uint32_t* p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.cta.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(smem_u32(p)), "r"(v) : "memory");
    return old;
}

// Thread-block cluster: barrier over all threads of all CTAs of the cluster (release / acquire), this
// CTA's rank, the address of a shared-memory location in another CTA of the cluster, and a load from it.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to_cluster_cta(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
// n / d for 0 <= n < 2^23 through the reciprocal inv = 1 / d (a handful of instructions where the
// integer division is a few dozen; the epilogue divides several times per output)
__device__ __forceinline__ int div_small(int n, int d, float inv) {
    int q = __float2int_rz(__int2float_rn(n) * inv);
    if (q * d > n) --q;
    else if ((q + 1) * d <= n) ++q;
    return q;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// Warps per CTA and with them the registers a thread may have (spmm_warps()).
template <int NT> constexpr int kWarpsOf = NT == 1 ? 32 : NT == 8 ? 8 : 16;

template <int MT, int NT>
__global__ void __launch_bounds__(kWarpsOf<NT> * 32, 1) csb_spmm_tile_kernel(const __grid_constant__ SpmmArgs a) {
    constexpr int kSpmmWarps = kWarpsOf<NT>;
    pdl_launch_dependents();
    extern __shared__ __align__(128) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const SpmmSmem L(kSpmmWarps, a.w_stages, a.x_depth, a.tile_bytes, a.pitch, MT, NT, spmm_q_bytes(NT, a.q_rows));
    uint64_t* wfull = reinterpret_cast<uint64_t*>(smem + L.wfull) + warp * a.w_stages;
    uint64_t* xfull = reinterpret_cast<uint64_t*>(smem + L.xfull);
    uint32_t* xcnt = reinterpret_cast<uint32_t*>(smem + L.xcnt);
    volatile uint32_t* s_dead = reinterpret_cast<volatile uint32_t*>(smem + L.dead);
    uint8_t* wring = smem + L.wring + (size_t)warp * a.w_stages * kSpmmStageBytes;
    uint8_t* xring = smem + L.xring;
    const uint32_t zero_addr = smem_u32(smem + L.zero);

#ifdef CSB_SPMM_CLOCKS
    long long sprof[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    long long st_ = clock64();
#endif
    // the CTA's descriptor goes to shared memory, one word per thread
    __shared__ __align__(16) SpmmCta s_me;
    __shared__ int s_first[5];                     // first warp of every block-row of the group (the warps of a row are neighbours)
    if (threadIdx.x == 0) {
        for (int i = 0; i < kSpmmWarps * a.w_stages; ++i) mbar_init(reinterpret_cast<uint64_t*>(smem + L.wfull) + i, 1);
        for (int i = 0; i < a.x_depth; ++i) { mbar_init(&xfull[i], 1); xcnt[i] = 0u; }
        *s_dead = 0u;
        mbar_fence_init();
    }
    for (int i = threadIdx.x; i < (a.pitch + 16) / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(smem + L.zero)[i] = 0u;
    int p_idx = 0, cta0 = 0;                       // which product this CTA works for, and its first CTA
    while (p_idx + 1 < a.n_parts && (int)blockIdx.x >= a.part[p_idx].cta_end) { cta0 = a.part[p_idx].cta_end; ++p_idx; }
    const SpmmPart& pt = a.part[p_idx];
    const int cta = (int)blockIdx.x - cta0;
    int xs = 0, s = 0;                             // slot of the input ring the warp is at; stage of its weight ring
    uint32_t xpar = 0u, parity = 0u;               // and the parities of their current uses
    // The first chunks of a warp's weight stream go out, into the stages in ring order; returns where the
    // next chunk to be fetched starts.  (A warp's chunks lie back to back.)
    auto first_weights = [&](const uint8_t* stream, const uint4& d) -> uint32_t {
        const uint32_t first[3] = {d.z & 0xffffu, d.z >> 16, d.w};
        uint32_t off = d.x;
        int si = s;
        for (int k = 0; k < a.w_stages && k < (int)d.y; ++k) {
            if (lane == 0) {
                mbar_expect_tx(&wfull[si], first[k]);
                bulk_g2s(wring + (size_t)si * kSpmmStageBytes, stream + (size_t)off * 16, first[k], &wfull[si]);
            }
            off += first[k] >> 4;
            if (++si == a.w_stages) si = 0;
        }
        return off;
    };
    if (threadIdx.x < sizeof(SpmmCta) / 4)
        reinterpret_cast<uint32_t*>(&s_me)[threadIdx.x] = reinterpret_cast<const uint32_t*>(pt.ctas + cta)[threadIdx.x];
    const uint4 wd = __ldg(pt.warp_desc + (size_t)cta * kSpmmWarps + warp);
    const uint32_t n_chunks = wd.y;
    __syncthreads();
    const SpmmCta* me = &s_me;
    const int ntiles = me->ntiles, tile0 = me->tile0;
    auto tile_bytes_of = [&](int tl) { return (uint32_t)min(a.tile_cols, pt.cols - (tile0 * a.block_c + tl * a.tile_cols)) * (uint32_t)a.pitch; };
    auto tile_src = [&](int tl) { return pt.xp + (size_t)(tile0 * a.block_c + tl * a.tile_cols) * a.pitch; };
    // the weights were written at plan time: their first copies go out before the work in front is waited for
    // (a warp's chunks lie back to back; issue_off is where the next one to be fetched starts)
    uint32_t issue_off = first_weights(pt.stream, wd);
    if (threadIdx.x == 0) {
        int rr = 0;
        s_first[0] = 0;
        for (int w = 0; w < kSpmmWarps; ++w)
            while (rr < (int)me->warp_row[w]) s_first[++rr] = w;
        while (rr < 4) s_first[++rr] = kSpmmWarps;
    }
    pdl_wait();                                    // the packed inputs and Y belong to the work in front on the stream
    // One lane fetches a tile with one bulk copy.  (No proxy fence in front of a refill: the slot's
    // readers have their data in registers by the time they release it, and the release orders them
    // before this copy is issued.)
    auto fetch_tile = [&](int slot, int tl) {
        if (lane == 0) {
            mbar_expect_tx(&xfull[slot], tile_bytes_of(tl));
            bulk_g2s(xring + (size_t)slot * a.tile_bytes, tile_src(tl), tile_bytes_of(tl), &xfull[slot]);
        }
    };
    if (warp < a.x_depth && warp < ntiles) fetch_tile((xs + warp) % a.x_depth, warp);     // the first tiles, one warp each
    SPMM_LAP(0);                                   // set-up, first copies out, the work in front waited for
    // A wait gives up after a second, or as soon as any warp of the CTA has given up.
    auto wait_bar = [&](uint64_t* bar, uint32_t parity) -> bool {
        bool ok = mbar_try_wait(bar, parity);
        if (!ok) {
            unsigned long long t0 = 0;                // the clock is a slow read: only every 256 failed polls
            unsigned int spins = 0;
            for (;;) {
                if (mbar_try_wait_parked(bar, parity, 4000u)) { ok = true; break; }
                if ((++spins & 255u) == 0) {
                    if (*s_dead) break;
                    const unsigned long long now = global_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > kCopyWaitNs) { *s_dead = 1u; *(volatile uint32_t*)a.status = (uint32_t)kDevCopyTimeout; break; }
                }
            }
        }
        return __all_sync(0xffffffffu, ok);          // the whole warp goes on, or none of it
    };
    // The tile this warp is at (tcur) sits in slot xs of the input ring, in the use of that slot with
    // parity xpar; both move along with tcur, so nothing is divided.
    int tcur = 0;
    auto wait_x = [&]() -> bool { return wait_bar(&xfull[xs], xpar); };
    // This warp is done with tile tcur; the last warp of the CTA to say so refills the slot.
    auto release_x = [&]() {
        __syncwarp();
        uint32_t last = 0u;
        // The add releases this warp's reads of the slot and, for the last warp, acquires the others' before its
        // copy overwrites the slot (a relaxed add would lean on the order in which the hardware happens to do a
        // warp's accesses to shared memory; 60.2 against 60.1 us, 8192 x 8192 at 4x, batch 64).
        if (lane == 0) {
            last = atom_add_acq_rel_shared(&xcnt[xs], 1u) == (uint32_t)kSpmmWarps - 1u;
            if (last) *reinterpret_cast<volatile uint32_t*>(&xcnt[xs]) = 0u;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last && tcur + a.x_depth < ntiles) fetch_tile(xs, tcur + a.x_depth);
        ++tcur;
        if (++xs == a.x_depth) { xs = 0; xpar ^= 1u; }
    };

    float acc[MT][NT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.f;

    const uint32_t x_lane_off = (uint32_t)(lane >> 4) * 16u;                 // this lane's 16 bytes inside a tile row
    const int kr_lane = ((lane >> 3) & 1) * 8 + (lane & 7);                  // its k row inside a 16-column slab
    bool alive = true;
    for (uint32_t c = 0; c < n_chunks && alive; ++c) {
        SPMM_LAP(4);
        if (!wait_bar(&wfull[s], parity)) { alive = false; break; }
        SPMM_LAP(1);                               // waiting for weights
        const uint8_t* p = wring + (size_t)s * kSpmmStageBytes;
        const uint4 chh = *reinterpret_cast<const uint4*>(p);              // items' size, sizes of the next three chunks
        const uint8_t* end = p + 16 + 16 * (size_t)chh.x;
        const uint32_t refill_bytes = a.w_stages == 3 ? chh.w : chh.z;     // the chunk w_stages further on
        p += 16;
        while (p < end) {
            const uint4 h = *reinterpret_cast<const uint4*>(p);
            const int tile = (int)(h.x & 0xffffu), nk = (int)((h.x >> 16) & 0xffu), np2 = (int)(h.x >> 24);
            const uint32_t mask_lo = h.y, mask_hi = h.z;
            const uint8_t* cidx = p + 16;
            const uint32_t vals = smem_u32(cidx + ((nk + 3) & ~3));
            p += 16 * (size_t)(h.w & 0xffffu);
            // tiles this warp has no block in are passed in order
            SPMM_LAP(4);
            while (tcur < tile && alive) {
                if (!wait_x()) { alive = false; break; }
                release_x();
            }
            if (!alive || !wait_x()) { alive = false; break; }
            SPMM_LAP(2);                           // passing tiles and waiting for this item's tile
            const uint32_t xtile = smem_u32(xring + (size_t)xs * a.tile_bytes);
            // address of this lane's words in the stored row behind each of its output rows (rows that are
            // not kept have none).  Lane l works out where in-block rows l and l + 32 are stored (a
            // population count on the row mask) and the lanes fetch what they need by shuffle.
            uint32_t rowaddr[MT][2];
            {
                const uint32_t below = (1u << lane) - 1u;
                const uint32_t e_lo = ((mask_lo >> lane) & 1u) ? (uint32_t)__popc(mask_lo & below) : 0xffffu;
                const uint32_t e_hi = ((mask_hi >> lane) & 1u) ? (uint32_t)(__popc(mask_lo) + __popc(mask_hi & below)) : 0xffffu;
                const uint32_t mine = e_lo | (e_hi << 16);
#pragma unroll
                for (int q = 0; q < (MT < 2 ? MT : 2); ++q)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const uint32_t v = __shfl_sync(0xffffffffu, mine, 16 * q + g + 8 * hh);
                        const uint32_t lo = v & 0xffffu, hi = v >> 16;
                        rowaddr[q][hh] = lo != 0xffffu ? vals + (lo * (uint32_t)np2 + (uint32_t)t) * 4u : kNoRow;
                        if (MT > 2) rowaddr[(q + 2) % MT][hh] = hi != 0xffffu ? vals + (hi * (uint32_t)np2 + (uint32_t)t) * 4u : kNoRow;
                    }
            }
            for (int kb = 0; kb < nk; kb += 16) {
                // ---- B operand: the gathered inputs, 16 kept columns x this warp's batch columns
                const int kr = kb + kr_lane;
                const uint32_t rowp = (kr < nk ? xtile + (uint32_t)cidx[kr] * (uint32_t)a.pitch : zero_addr) + x_lane_off;
                uint32_t bh[NT][2], bl[NT][2];
                if (NT == 1) {
                    uint32_t r4[4];
                    ldmatrix_x4_trans(r4, rowp);                       // (hi, k 0-7), (hi, k 8-15), (lo, k 0-7), (lo, k 8-15)
                    bh[0][0] = r4[0]; bh[0][1] = r4[1]; bl[0][0] = r4[2]; bl[0][1] = r4[3];
                } else {
#pragma unroll
                    for (int q = 0; q < NT / 2; ++q) {
                        uint32_t r4[4];
                        ldmatrix_x4_trans(r4, rowp + 32u * q);         // batch tiles 2q, 2q + 1 of the hi part
                        bh[2 * q][0] = r4[0]; bh[2 * q][1] = r4[1]; bh[(2 * q + 1) % NT][0] = r4[2]; bh[(2 * q + 1) % NT][1] = r4[3];
                        ldmatrix_x4_trans(r4, rowp + 16u * NT + 32u * q);   // the same of the lo part
                        bl[2 * q][0] = r4[0]; bl[2 * q][1] = r4[1]; bl[(2 * q + 1) % NT][0] = r4[2]; bl[(2 * q + 1) % NT][1] = r4[3];
                    }
                }
                // ---- A operand: the kernel matrix with its rows at their RowIdx positions.  Words past the
                // end of a stored row (last slab of a slice that is not a multiple of 16 wide) are zero.
                const uint32_t koff = (uint32_t)kb * 2u;                             // bytes into a stored row
                const bool v0 = (uint32_t)(kb >> 1) + (uint32_t)t < (uint32_t)np2, v1 = (uint32_t)(kb >> 1) + (uint32_t)t + 4u < (uint32_t)np2;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    uint32_t af[4];
                    af[0] = (rowaddr[mt][0] != kNoRow && v0) ? lds_u32(rowaddr[mt][0] + koff) : 0u;
                    af[1] = (rowaddr[mt][1] != kNoRow && v0) ? lds_u32(rowaddr[mt][1] + koff) : 0u;
                    af[2] = (rowaddr[mt][0] != kNoRow && v1) ? lds_u32(rowaddr[mt][0] + koff + 16u) : 0u;
                    af[3] = (rowaddr[mt][1] != kNoRow && v1) ? lds_u32(rowaddr[mt][1] + koff + 16u) : 0u;
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        mma_m16n8k16(acc[mt][nt], af, bh[nt][0], bh[nt][1]);
                        mma_m16n8k16(acc[mt][nt], af, bl[nt][0], bl[nt][1]);
                    }
                }
            }
            SPMM_LAP(3);                           // row map, operand loads, tensor instructions
        }
        if (!alive) break;
        // this warp is done with the stage and refills it
        __syncwarp();
        if (refill_bytes) {
            if (lane == 0) {
                mbar_expect_tx(&wfull[s], refill_bytes);
                bulk_g2s(wring + (size_t)s * kSpmmStageBytes, pt.stream + (size_t)issue_off * 16, refill_bytes, &wfull[s]);
            }
            issue_off += refill_bytes >> 4;
        }
        if (++s == a.w_stages) { s = 0; parity ^= 1u; }
    }
    SPMM_LAP(4);                                   // ring bookkeeping
    while (tcur < ntiles && alive) {
        if (!wait_x()) { alive = false; break; }
        release_x();
    }
    SPMM_LAP(5);                                   // the tiles behind this warp's last item
    __syncthreads();
    SPMM_LAP(6);                                   // waiting for the other warps of the CTA
    const bool dead = *s_dead != 0u;
    if (dead) {
        // a wait gave up (the status word says so): give copies that may still be in flight a bounded
        // time to land before the CTA's shared memory goes away, and write nothing
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        if (a.S == 1) return;                      // (a CTA of a cluster still has to keep the cluster's barriers company)
    }

    // ---- the warps' sums meet in shared memory (the rings are no longer in use)
    constexpr int kP = spmm_sum_pitch(NT);
    float* P = reinterpret_cast<float*>(smem + L.rings);           // [warp][row of the block][kP]
    {
        float* Pw = P + (size_t)warp * MT * 16 * kP;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float* q = Pw + (16 * mt + g) * kP + 8 * nt + 2 * t;
                *reinterpret_cast<float2*>(q) = make_float2(acc[mt][nt][0], acc[mt][nt][1]);
                *reinterpret_cast<float2*>(q + 8 * kP) = make_float2(acc[mt][nt][2], acc[mt][nt][3]);
            }
    }
    __syncthreads();
    SPMM_LAP(7);                                   // accumulators to shared memory
    const int group_rows = pt.RG * a.block_r, row0 = me->group * group_rows;
    const int nrows = min(group_rows, pt.rows - row0);
    // this CTA's sums over its range: [batch column][row of the group], one float of padding per column
    // (written four columns at a time without bank conflicts, read by the cluster in runs of consecutive rows)
    float* part = reinterpret_cast<float*>(smem + L.qsums);
    const int kQ = group_rows + 1;
    {
        // one thread per row and four batch columns; the warps of a block-row are added in warp order
        constexpr int kQuads = 2 * NT;
        const int total = dead ? 0 : nrows * kQuads;
        const float inv_br = 1.f / (float)a.block_r;
        // (four of a thread's outputs at a time, so that their loads are in flight together)
        for (int i0 = threadIdx.x; i0 < total; i0 += 4 * blockDim.x) {
            const float* src[4];
            int cnt[4], rl[4], q4[4], cmax = 0;
            float4 sum[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = min(i0 + j * (int)blockDim.x, total - 1);
                rl[j] = i / kQuads; q4[j] = i % kQuads;
                const int rr = div_small(rl[j], a.block_r, inv_br), rin = rl[j] - rr * a.block_r;
                const int w0 = s_first[rr];
                cnt[j] = s_first[rr + 1] - w0;
                cmax = max(cmax, cnt[j]);
                src[j] = P + ((size_t)w0 * MT * 16 + rin) * kP + 4 * q4[j];
                sum[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            for (int k = 0; k < cmax; ++k) {
                float4 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = k < cnt[j] ? *reinterpret_cast<const float4*>(src[j] + (size_t)k * MT * 16 * kP) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 4; ++j) { sum[j].x += v[j].x; sum[j].y += v[j].y; sum[j].z += v[j].z; sum[j].w += v[j].w; }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j * (int)blockDim.x < total) {
                    float* dst = part + 4 * q4[j] * kQ + rl[j];
                    dst[0] = sum[j].x; dst[kQ] = sum[j].y; dst[2 * kQ] = sum[j].z; dst[3 * kQ] = sum[j].w;
                }
        }
    }
    __syncthreads();
    SPMM_LAP(8);                                   // sums over the warps of a block-row
    // The S CTAs of a row group form a thread-block cluster.  Once all of them have their sums in shared
    // memory, every CTA adds up the S ranges, in range order, for its share of the group's rows, reading
    // the other CTAs' sums through distributed shared memory; nobody leaves before everybody has read.
    // (The CTA barriers in front keep each warp together for the aligned cluster barrier.)
    if (a.S > 1) cluster_barrier();
    SPMM_LAP(9);                                   // waiting for the cluster's other CTAs
    {
        const uint32_t rank = a.S > 1 ? cluster_rank() : 0u;
        const int share = (nrows + a.S - 1) / a.S, r_lo = min(nrows, (int)rank * share), r_n = min(nrows, r_lo + share) - r_lo;
        const uint32_t q_local = smem_u32(part);
        uint32_t q_of[8];
#pragma unroll
        for (int s2 = 0; s2 < 8; ++s2) q_of[s2] = a.S > 1 && s2 < a.S ? map_to_cluster_cta(q_local, (uint32_t)s2) : q_local;
        // a warp takes batch columns, its lanes consecutive rows: stores of 128 contiguous bytes
        // (two batch columns x two runs of rows per lane at a time: up to 32 remote loads in flight)
        for (int b0 = warp; b0 < (dead ? 0 : a.nb); b0 += 2 * kSpmmWarps)
            for (int r0 = lane; r0 < r_n; r0 += 64) {
                float v[4][8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int b = b0 + (j >> 1) * kSpmmWarps, r = r0 + (j & 1) * 32;
                    const bool live = b < a.nb && r < r_n;
                    const uint32_t off = (uint32_t)(b * kQ + r_lo + r) * 4u;
#pragma unroll
                    for (int s2 = 0; s2 < 8; ++s2) {
                        if (a.S > 1) v[j][s2] = live && s2 < a.S ? ld_cluster_f32(q_of[s2] + off) : 0.f;
                        else v[j][s2] = live && s2 == 0 ? part[b * kQ + r_lo + r] : 0.f;
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int b = b0 + (j >> 1) * kSpmmWarps, r = r0 + (j & 1) * 32;
                    float sum = v[j][0];
#pragma unroll
                    for (int s2 = 1; s2 < 8; ++s2) sum += v[j][s2];
                    if (b < a.nb && r < r_n) pt.Y[(long long)b * a.ldy + row0 + r_lo + r] = sum;
                }
            }
    }
    SPMM_LAP(10);                                  // sums over the ranges, store
    if (a.S > 1) {
        __syncthreads();
        cluster_barrier();
    }
    SPMM_LAP(11);                                  // until every CTA of the cluster has read
#ifdef CSB_SPMM_CLOCKS
    if (lane == 0) for (int i = 0; i < 16; ++i) a.clocks[((size_t)blockIdx.x * kSpmmWarps + warp) * 16 + i] = sprof[i];
#endif
}

#define CSB_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            set_error("%s failed: %s", #call, cudaGetErrorString(e_));                     \
            return e_ == cudaErrorMemoryAllocation ? CSB_ERR_ALLOC : CSB_ERR_CUDA;         \
        }                                                                                  \
    } while (0)

bool spmm_mma_applicable(const csb_matrix* A, int batch) {
    if (getenv("CSB_NO_MMA") && atoi(getenv("CSB_NO_MMA"))) return false;
    if (!(batch >= 8 && A->val_dtype == CSB_F16 && A->block_r <= 64 && A->device >= 0)) return false;
    return !(A->mma && A->mma->cls[spmm_class_index(batch)].unusable);
}

template <typename V>
static int upload_v(const std::vector<V>& h, V** d) {
    const size_t bytes = std::max<size_t>(h.size(), 1) * sizeof(V);
    CSB_CUDA(cudaMalloc((void**)d, bytes));
    if (!h.empty()) CSB_CUDA(cudaMemcpy(*d, h.data(), h.size() * sizeof(V), cudaMemcpyHostToDevice));
    return CSB_OK;
}

static int mt_of(const csb_matrix* A) { return A->block_r <= 16 ? 1 : A->block_r <= 32 ? 2 : 4; }

template <int MT, int NT> struct SetSmem {
    static cudaError_t call(size_t bytes) { return cudaFuncSetAttribute(csb_spmm_tile_kernel<MT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); }
};
template <int MT, int NT> struct MaxClusters {
    static cudaError_t call(int* n, const cudaLaunchConfig_t* cfg) { return cudaOccupancyMaxActiveClusters(n, csb_spmm_tile_kernel<MT, NT>, cfg); }
};
template <int MT, int NT> struct LaunchTile {
    static cudaError_t call(const cudaLaunchConfig_t* cfg, const SpmmArgs& a) { return cudaLaunchKernelEx(cfg, csb_spmm_tile_kernel<MT, NT>, a); }
};
template <template <int, int> class F, int MT, typename... X>
static cudaError_t spmm_dispatch_nt(int NT, X&&... x) {
    return NT == 1 ? F<MT, 1>::call(x...) : NT == 2 ? F<MT, 2>::call(x...) : NT == 4 ? F<MT, 4>::call(x...) : F<MT, 8>::call(x...);
}
template <template <int, int> class F, typename... X>
static cudaError_t spmm_dispatch(int MT, int NT, X&&... x) {
    return MT == 1 ? spmm_dispatch_nt<F, 1>(NT, x...) : MT == 2 ? spmm_dispatch_nt<F, 2>(NT, x...) : spmm_dispatch_nt<F, 4>(NT, x...);
}

// Room for packed inputs: whole tiles, so that a tile copy never runs past the end.
static int alloc_packed(const csb_matrix* A, int NT, MmaPlan::PerClass* P) {
    const size_t bytes = (size_t)A->nbc * A->block_c * spmm_pitch(NT);
    CSB_CUDA(cudaMalloc(&P->d_xp, bytes));
    CSB_CUDA(cudaMemset(P->d_xp, 0, bytes));
    return CSB_OK;
}

// The plan of A for batch tiles of 8 * NT columns on `sms` SMs; force_S > 0 fixes the cluster size (the products of
// one launch share it).
static int build_spmm_plan(const csb_matrix* A, int ci, int sms, int force_S, bool with_x, MmaPlan::PerClass* P) {
    const int NT = 1 << ci;
    SpmmHostPlan H;
    int rc = plan_spmm_host(A, NT, sms, force_S, &H);
    if (rc == 1) { P->unusable = true; return CSB_OK; }
    if (rc != CSB_OK) return rc;
    const int MT = mt_of(A), pitch = spmm_pitch(NT);
    const int tile_bytes = (spmm_tile_blocks(A->block_c) * A->block_c * pitch + 127) & ~127;
    // rings: as many weight stages (3, else 2) and input tiles (up to 8, at least 2) as shared memory holds
    int w_stages = 0, x_depth = 0;
    size_t smem = 0;
    for (int ws = 3; ws >= 2 && !x_depth; --ws)
        for (int xd = std::min(8, std::max(2, H.max_tiles)); xd >= 2; --xd) {
            const SpmmSmem L(spmm_warps(NT), ws, xd, tile_bytes, pitch, MT, NT, spmm_q_bytes(NT, H.RG * A->block_r));
            if (L.total + kSpmmStaticSmem <= A->smem_optin) { w_stages = ws; x_depth = xd; smem = L.total; break; }
        }
    if (!x_depth) { P->unusable = true; return CSB_OK; }
    P->RG = H.RG; P->S = H.S; P->n_ctas = (int)H.ctas.size(); P->n_groups = H.n_groups;
    P->w_stages = w_stages; P->x_depth = x_depth; P->smem_bytes = smem; P->balance = H.balance; P->warp_balance = H.warp_balance;
    P->stream_bytes = (int64_t)H.bytes.size();
    if ((rc = upload_v(H.bytes, &P->d_stream)) != CSB_OK) return rc;
    if ((rc = upload_v(H.warp_desc, &P->d_warp_desc)) != CSB_OK) return rc;
    if ((rc = upload_v(H.ctas, &P->d_ctas)) != CSB_OK) return rc;
    if (with_x && (rc = alloc_packed(A, NT, P)) != CSB_OK) return rc;
    // (the limit belongs to the kernel, not to this plan: other matrices launch the same instantiation with other sizes)
    CSB_CUDA(spmm_dispatch<SetSmem>(MT, NT, A->smem_optin - kSpmmStaticSmem));
    if (H.S > 1) {
        // the S CTAs of a row group are launched as one cluster: make sure such a cluster can be resident
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)H.S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)H.ctas.size()); cfg.blockDim = dim3((unsigned)spmm_warps(NT) * 32u); cfg.dynamicSmemBytes = smem;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int clusters = 0;
        CSB_CUDA(spmm_dispatch<MaxClusters>(MT, NT, &clusters, &cfg));
        if (clusters < 1) { P->unusable = true; return CSB_OK; }
    }
    CSB_CUDA(cudaDeviceSynchronize());
    P->built = true;
    return CSB_OK;
}

static void drop_plan(MmaPlan::PerClass& c) {
    cudaFree(c.d_stream); cudaFree(c.d_warp_desc); cudaFree(c.d_ctas); cudaFree(c.d_xp);
    c.d_stream = nullptr; c.d_warp_desc = nullptr; c.d_ctas = nullptr; c.d_xp = nullptr;
}
void free_mma(csb_matrix* A) {
    if (!A->mma) return;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(A->device);
    for (auto& c : A->mma->cls) drop_plan(c);
    for (auto& c : A->mma->shared) drop_plan(c.plan);
    drop_umma_plan(A->mma->umma);
    cudaSetDevice(prev);
    delete A->mma;
    A->mma = nullptr;
}

#ifdef CSB_SPMM_CLOCKS
static long long* g_spmm_clocks = nullptr;
static int g_spmm_clock_warps = 0;
extern "C" int csb_debug_spmm_clocks(long long* host_out, int max_warps) {
    cudaMemcpy(host_out, g_spmm_clocks, (size_t)std::min(max_warps, g_spmm_clock_warps) * 16 * 8, cudaMemcpyDeviceToHost);
    return g_spmm_clock_warps;
}
#endif

static int make_spmm_plan(const csb_matrix* A, int ci, int sms, int force_S, bool with_x, MmaPlan::PerClass* C) {
    if (!C->built && !C->unusable) {
        int rc;
        try { rc = build_spmm_plan(A, ci, sms, force_S, with_x, C); }
        catch (const std::bad_alloc&) { set_error("out of host memory while planning the batched product"); rc = CSB_ERR_ALLOC; }
        if (rc != CSB_OK) {                                // (what it had allocated goes back, and no error is left behind for the next launch to find)
            drop_plan(*C);
            cudaGetLastError();
            C->unusable = true;
            return rc;
        }
    }
    return (C->unusable || !C->built) ? 1 : CSB_OK;
}
static int ensure_mma(const csb_matrix* A) {
    if (!A->mma) A->mma = new (std::nothrow) MmaPlan();
    if (A->mma) return CSB_OK;
    set_error("out of host memory");
    return CSB_ERR_ALLOC;
}

// Launches the tile kernel over the products (P[i], xp[i], Y[i]) of matrices with the same block shape.
static int launch_parts(int n, const csb_matrix* const* A, const MmaPlan::PerClass* const* P, const uint8_t* const* xp, float* const* Y, int NT, int nb,
                        int64_t ldy, cudaStream_t st) {
    note_tensor_kernel(kTensorMma);
    const int MT = mt_of(A[0]);
    SpmmArgs a{};
    a.n_parts = n; a.nb = nb; a.ldy = ldy; a.status = A[0]->product.d_status;
    a.block_r = A[0]->block_r; a.block_c = A[0]->block_c; a.S = P[0]->S;
    a.tile_cols = spmm_tile_blocks(a.block_c) * a.block_c;
    a.pitch = spmm_pitch(NT); a.tile_bytes = (a.tile_cols * a.pitch + 127) & ~127;
    a.x_depth = P[0]->x_depth; a.w_stages = P[0]->w_stages;
    int ctas = 0;
    for (int i = 0; i < n; ++i) {
        SpmmPart& p = a.part[i];
        p.stream = P[i]->d_stream; p.warp_desc = (const uint4*)P[i]->d_warp_desc; p.ctas = P[i]->d_ctas; p.xp = xp[i]; p.Y = Y[i];
        p.rows = (int)A[i]->rows; p.cols = (int)A[i]->cols; p.RG = P[i]->RG;
        ctas += P[i]->n_ctas;
        p.cta_end = ctas;
        a.x_depth = std::min(a.x_depth, P[i]->x_depth); a.w_stages = std::min(a.w_stages, P[i]->w_stages);
        a.q_rows = std::max(a.q_rows, P[i]->RG * a.block_r);
    }
    const SpmmSmem L(spmm_warps(NT), a.w_stages, a.x_depth, a.tile_bytes, a.pitch, MT, NT, spmm_q_bytes(NT, a.q_rows));
#ifdef CSB_SPMM_CLOCKS
    if (!g_spmm_clocks) cudaMalloc((void**)&g_spmm_clocks, (size_t)1 << 24);
    a.clocks = g_spmm_clocks;
    g_spmm_clock_warps = ctas * spmm_warps(NT);
#endif
    // the kernel orders itself behind the work in front (pdl_wait), so it may be launched with programmatic
    // stream serialization: its scheduling overlaps that work's tail
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;             // the CTAs that share a row group
    attr[1].val.clusterDim.x = (unsigned)a.S; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = a.S > 1 ? 2 : 1;
    cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3((unsigned)spmm_warps(NT) * 32u); cfg.dynamicSmemBytes = L.total;
    CSB_CUDA(spmm_dispatch<LaunchTile>(MT, NT, &cfg, a));
    CSB_CUDA(cudaGetLastError());
    return CSB_OK;
}

// Packs fp32 inputs into `xp` and launches, 8 * NT batch columns at a time.
static int pack_and_launch(const csb_matrix* A, const MmaPlan::PerClass* P, int NT, uint8_t* xp, const float* X, int64_t ldx, int batch, float* Y,
                           int64_t ldy, cudaStream_t st) {
    const int cap = 8 * NT;
    for (int b0 = 0; b0 < batch; b0 += cap) {
        const int nb = std::min(cap, batch - b0);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 1;
        cfg.gridDim = dim3((unsigned)((A->cols + 31) / 32)); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = 0;
        CSB_CUDA(cudaLaunchKernelEx(&cfg, csb_pack_x_kernel, X + (int64_t)b0 * ldx, (long long)ldx, nb, (int)A->cols, xp, spmm_pitch(NT), NT));
        const uint8_t* packed = xp;
        float* y = Y + (int64_t)b0 * ldy;
        const int rc = launch_parts(1, &A, &P, &packed, &y, NT, nb, ldy, st);
        if (rc != CSB_OK) return rc;
    }
    return CSB_OK;
}

static bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &status) != cudaSuccess) { cudaGetLastError(); return false; }
    return status != cudaStreamCaptureStatusNone;
}

// Returns CSB_OK after launching, or 1 when the caller should use the CUDA-core path.
int launch_spmm_mma(const csb_matrix* A, const float* X, int64_t ldx, int batch, float* Y, int64_t ldy, void* stream) {
    int rc = product_gave_up(A);
    if (rc != CSB_OK) return rc;
    int prev = 0;
    CSB_CUDA(cudaGetDevice(&prev));
    if (prev != A->device) CSB_CUDA(cudaSetDevice(A->device));
    struct Restore { int prev, cur; ~Restore() { if (prev != cur) cudaSetDevice(prev); } } restore{prev, A->device};
    if (umma_applicable(A)) {
        std::lock_guard<std::mutex> lk(A->mma_mu);
        if ((rc = ensure_mma(A)) != CSB_OK) return rc;
        if ((rc = launch_umma(A, &A->mma->umma, X, ldx, batch, Y, ldy, stream)) != 1) return rc;
        clear_error();
    }
    // Eight columns run in tiles of 16: half as many warps with twice the columns meet at half as many hand-overs, and
    // the columns of zeros cost less than that (8 x 32-warp tiles against these, us: 3072 x 1536 at 8x 13.0 / 10.5, 4096 x
    // 4096 of 32 x 32 blocks at 5x 24.0 / 15.5, 8192 x 8192 at 4x 28.2 / 27.5; the one that lost, 4096 x 4096 of
    // 64 x 64 blocks at 5x, 13.7 / 14.1).  The recurrent stacks keep tiles of 8, their plans share a grid.
    int ci = std::max(1, spmm_class_index(batch));
    const int sms = A->opts.ctas > 0 ? A->opts.ctas : A->sm_count;
    {
        std::lock_guard<std::mutex> lk(A->mma_mu);
        if ((rc = ensure_mma(A)) != CSB_OK) return rc;
        MmaPlan::PerClass* cls = A->mma->cls;
        // more than 32 columns: tiles of 64, so that row maps, weights and bookkeeping are paid once for all of
        // them (8192 x 8192 at 4x, batch 64: 74.9 -> 59.3 us); where that plan does not fit, passes of 32
        if (batch > 32) ci = 3;
        // either of the two wide layouts serves any batch: in a stream capture, where none can be built, the one there is
        if (ci >= 2 && !cls[ci].built && cls[5 - ci].built && capturing((cudaStream_t)stream)) ci = 5 - ci;
        if (ci == 3 && make_spmm_plan(A, 3, sms, 0, true, &cls[3]) != CSB_OK) { clear_error(); ci = 2; }
        rc = make_spmm_plan(A, ci, sms, 0, true, &cls[ci]);
        if (rc == 1 && batch <= 8) rc = make_spmm_plan(A, ci = 0, sms, 0, true, &cls[0]);   // takes less shared memory
        if (rc != CSB_OK) return rc;
    }
    const MmaPlan::PerClass* P = &A->mma->cls[ci];
    return pack_and_launch(A, P, 1 << ci, (uint8_t*)P->d_xp, X, ldx, batch, Y, ldy, (cudaStream_t)stream);
}

// The products of a stack's layers over inputs packed by the caller (one row of spmm_pitch(NT) bytes per matrix
// column: the hi parts of 8 * NT batch slots, then the lo parts), at most 32 batch columns.  Prepared once
// per stack: the SMs are shared between the layers in proportion to their weights when the layers' blocks
// have the same shape and one launch can hold all of them (*joint = true), else every layer has all of them.
int prepare_spmm_stack(int L, const csb_matrix* const* A, int batch, SpmmStack* out) {
    const int ci = spmm_class_index(batch);
    *out = SpmmStack{};
    out->NT = 1 << ci; out->L = L;
    bool joint = L > 1 && L <= kMaxLayers;
    int64_t nnz = 0;
    for (int l = 0; l < L; ++l) {
        joint = joint && A[l]->block_r == A[0]->block_r && A[l]->block_c == A[0]->block_c && A[l]->nnz > 0;
        nnz += A[l]->nnz;
    }
    const int sms = A[0]->opts.ctas > 0 ? A[0]->opts.ctas : A[0]->sm_count;
    int S = 0;
    // (the first layer's plan fixes the cluster size for all; layers above the first have the same shape)
    for (int pass = joint ? 0 : 1; pass < 2; ++pass) {
        bool fits = true;
        for (int l = L - 1; l >= 0 && fits; --l) {
            const int share = pass == 0 ? std::max(1, (int)(sms * (double)A[l]->nnz / (double)nnz)) : sms, want_S = pass == 0 ? S : 0;
            std::lock_guard<std::mutex> lk(A[l]->mma_mu);
            int rc = ensure_mma(A[l]);
            if (rc != CSB_OK) return rc;
            MmaPlan::PerClass* C = nullptr;
            for (auto& q : A[l]->mma->shared) if (q.ci == ci && q.sms == share && q.S == want_S) C = &q.plan;
            if (!C) {
                A[l]->mma->shared.push_back({ci, share, want_S, {}});
                C = &A[l]->mma->shared.back().plan;
            }
            rc = make_spmm_plan(A[l], ci, share, want_S, false, C);
            if (rc == 1) fits = false;
            else if (rc != CSB_OK) return rc;
            else { out->plan[l] = C; if (pass == 0 && S == 0) S = C->S; }
        }
        if (fits) { out->joint = pass == 0; return CSB_OK; }
    }
    return 1;
}

int launch_spmm_stack_fp32(const SpmmStack& K, int l, const csb_matrix* A, uint8_t* xp, const float* X, int64_t ldx, int batch, float* Y, int64_t ldy,
                           void* stream) {
    return pack_and_launch(A, K.plan[l], K.NT, xp, X, ldx, batch, Y, ldy, (cudaStream_t)stream);
}

int launch_spmm_stack(const SpmmStack& K, int l0, int l1, const csb_matrix* const* A, uint8_t* const* xp, float* const* Y, int nb, int64_t ldy, void* stream) {
    const uint8_t* x[kMaxLayers];
    for (int l = l0; l < l1; ++l) {
        const int rc = product_gave_up(A[l]);
        if (rc != CSB_OK) return rc;
        x[l] = xp[l];
    }
    if (K.joint) return launch_parts(l1 - l0, A + l0, K.plan + l0, x + l0, Y + l0, K.NT, nb, ldy, (cudaStream_t)stream);
    for (int l = l0; l < l1; ++l) {
        const int rc = launch_parts(1, A + l, K.plan + l, x + l, Y + l, K.NT, nb, ldy, (cudaStream_t)stream);
        if (rc != CSB_OK) return rc;
    }
    return CSB_OK;
}

}  // namespace csb

// Inspection / testing aid: the plan of the batched product, made on the host only.
extern "C" int csb_spmm_plan_dump(const csb_matrix_t* A, int batch, int sm_count, int64_t* info_out, uint8_t* stream_out, int64_t stream_cap,
                                  uint32_t* chunks_out, int64_t chunks_cap, uint32_t* stream_begin_out, int64_t begin_cap, int32_t* cta_out,
                                  int64_t cta_cap) {
    using namespace csb;
    clear_error();
    if (!A || !info_out || batch < 1 || sm_count < 1) { set_error("csb_spmm_plan_dump: bad argument"); return CSB_ERR_INVALID_ARG; }
    const int NT = batch > 32 ? 8 : spmm_nt(batch);
    SpmmHostPlan H;
    int rc;
    try { rc = plan_spmm_host(A, NT, sm_count, 0, &H); }
    catch (const std::bad_alloc&) { set_error("out of host memory while planning"); return CSB_ERR_ALLOC; }
    if (rc == 1) { set_error("the tensor-core layout does not apply to this matrix (fp16 values, block_r <= 64)"); return CSB_ERR_UNSUPPORTED; }
    if (rc != CSB_OK) return rc;
    info_out[0] = (int64_t)H.ctas.size(); info_out[1] = (int64_t)H.chunks.size(); info_out[2] = (int64_t)H.bytes.size();
    info_out[3] = H.RG; info_out[4] = NT | (spmm_warps(NT) << 8) | (spmm_tile_blocks(A->block_c) << 16); info_out[5] = H.S; info_out[6] = (int64_t)(H.warp_balance * 1e6);
    info_out[7] = (int64_t)(H.balance * 1e6);
    if (stream_out) {
        if (stream_cap < (int64_t)H.bytes.size()) { set_error("stream buffer too small"); return CSB_ERR_INVALID_ARG; }
        std::memcpy(stream_out, H.bytes.data(), H.bytes.size());
    }
    if (chunks_out) {
        if (chunks_cap < (int64_t)H.chunks.size()) { set_error("chunk buffer too small"); return CSB_ERR_INVALID_ARG; }
        for (size_t i = 0; i < H.chunks.size(); ++i) { chunks_out[2 * i] = H.chunks[i].off16; chunks_out[2 * i + 1] = H.chunks[i].bytes; }
    }
    if (stream_begin_out) {
        if (begin_cap < (int64_t)H.stream_begin.size()) { set_error("stream table too small"); return CSB_ERR_INVALID_ARG; }
        for (size_t i = 0; i < H.stream_begin.size(); ++i) stream_begin_out[i] = H.stream_begin[i];
    }
    if (cta_out) {
        if (cta_cap < (int64_t)H.ctas.size()) { set_error("CTA table too small"); return CSB_ERR_INVALID_ARG; }
        std::memcpy(cta_out, H.ctas.data(), H.ctas.size() * sizeof(SpmmCta));
    }
    return CSB_OK;
}
