// Host side of the batched product on tcgen05 tensor cores (csb_umma_kernel.cuh): packing and launches.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <mutex>

#include "csb_umma_rnn.hpp"
#include "csb_umma_kernel.cuh"

namespace csb {

// Packs fp32 inputs [nb][cols] into the operand images: one CTA per window, a thread per batch column and 8 matrix columns.
template <int NB>
__global__ void __launch_bounds__(NB * 8) csb_umma_pack_kernel(const float* __restrict__ X, long long ldx, int nb, int cols, int vec, uint8_t* __restrict__ xp,
                                                               uint32_t* __restrict__ bad) {
    pdl_launch_dependents();
    pdl_wait();                                           // X may come from the kernel in front; xp may still be read by it
    const int b = threadIdx.x >> 3, c = (int)blockIdx.x * kUmmaWindow + (threadIdx.x & 7) * 8;
    bool large = false;
    if (b < nb && c + 8 <= cols) large = put_eight<NB>(xp, b, c, cols, X + (long long)b * ldx + c, vec != 0);
    else {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = b < nb && c + i < cols ? X[(long long)b * ldx + c + i] : 0.f;
        large = put_split<NB>(xp, b, c, x);
    }
    large = __any_sync(0xffffffffu, large);
    if ((threadIdx.x & 31) == 0) bad[blockIdx.x * (NB / 4) + (threadIdx.x >> 5)] = large;
}

#define CSB_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            set_error("%s failed: %s", #call, cudaGetErrorString(e_));                     \
            return e_ == cudaErrorMemoryAllocation ? CSB_ERR_ALLOC : CSB_ERR_CUDA;         \
        }                                                                                  \
    } while (0)

template <int MODE>
static const void* pick_mode(int NB, int MT) {
    if (MT == 1) return NB == 16 ? (const void*)csb_umma_kernel<16, 1, MODE> : (const void*)csb_umma_kernel<32, 1, MODE>;
    return NB == 16 ? (const void*)csb_umma_kernel<16, 2, MODE> : (const void*)csb_umma_kernel<32, 2, MODE>;
}
// mode: 0 a product, 1 and 2 the time loops of LSTM and GRU (up to 32 batch columns)
const void* pick_umma(int mode, int NB, int MT) {
    if (mode == 1) return pick_mode<1>(NB, MT);
    if (mode == 2) return pick_mode<2>(NB, MT);
    if (NB < 64) return pick_mode<0>(NB, MT);
    return MT == 1 ? (const void*)csb_umma_kernel<64, 1, 0> : (const void*)csb_umma_kernel<64, 2, 0>;
}
// Stages of inputs, and what is left of `room` bytes of shared memory for values, in rounds of up to max_round bytes; false: too
// little.  (All of the room: a CTA takes all of TMEM, so two must not meet on an SM.)
bool umma_stages(int mode, int NB, int MT, int max_round, size_t room, UmmaStages* out) {
    for (int xd = x_windows(NB, MT) * NB * 256 >= 32768 ? 3 : kMaxXDepth; xd >= 2; --xd) {
        const UmmaSmem none(mode, NB, MT, xd, 0);
        const size_t fixed = (size_t)none.total - none.bars + none.w + (mode ? none.bars - none.part : 0);
        if (fixed >= room) continue;
        const int bytes = (int)((room - fixed) & ~(size_t)1023);
        if (bytes < (xd > 2 ? 2 : 1) * max_round || UmmaSmem(mode, NB, MT, xd, bytes).total > room) continue;
        *out = UmmaStages{xd, bytes, room};
        return true;
    }
    return false;
}

static cudaLaunchConfig_t umma_config(int ctas, int S, size_t smem, cudaStream_t st, cudaLaunchAttribute (&attr)[2]) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)S; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3(kUmmaThreads); cfg.dynamicSmemBytes = smem;
    cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = S > 1 ? 2 : 1;
    return cfg;
}

// Clusters of S CTAs that the device holds at a time, S = 1 .. kUmmaMaxS (SMs that a processing cluster's size leaves over
// are lost: 4 x 37 SMs do not make 37 clusters of four).
int umma_clusters(const csb_matrix* A, int (&n)[kUmmaMaxS + 1]) {
    const int sms = A->opts.ctas > 0 ? std::min(A->opts.ctas, A->sm_count) : A->sm_count;
    n[0] = 0; n[1] = sms;
    const void* kernel = pick_umma(0, 64, 2);
    const size_t smem = A->smem_optin;                     // (one CTA an SM in any case)
    CSB_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A->smem_optin));
    for (int S = 2; S <= kUmmaMaxS; ++S) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = umma_config(S * sms, S, smem, 0, attr);
        CSB_CUDA(cudaOccupancyMaxActiveClusters(&n[S], kernel, &cfg));
        n[S] = std::min(n[S], sms / S);
    }
    return CSB_OK;
}

int umma_nb(int batch) { return batch <= 16 ? 16 : batch <= 32 ? 32 : 64; }

static uint32_t* bad_words(uint8_t* xp, int windows) { return reinterpret_cast<uint32_t*>(xp + (size_t)windows * kUmmaImage); }

// Y = A . (packed inputs) with the plan's output rows.
int launch_umma_packed(const csb_matrix* A, const UmmaPlan* P, uint8_t* xp, float* Y, int NB, int nb, int64_t ldy, cudaStream_t st) {
    note_tensor_kernel(kTensorTiles);
    UmmaArgs a{};
    a.n_parts = 1; a.nb = nb; a.ldy = ldy; a.status = A->product.d_status; a.S = P->S; a.flush = P->flush;
    UmmaPart& p = a.part[0];
    UmmaStages g;
    if (!umma_stages(0, NB, P->MT, P->max_round, A->smem_optin, &g)) { set_error("the batched product's stages do not fit"); return CSB_ERR_LAUNCH; }
    a.x_depth = g.x_depth; a.w_bytes = g.w_bytes;
    p.stream = P->d_stream; p.ctas = P->d_ctas; p.rounds = P->d_rounds; p.quads = P->d_quads; p.xp = xp; p.bad = bad_words(xp, P->windows); p.Y = Y;
    p.block_r = A->block_r; p.seg_words = P->seg_words; p.windows = P->windows; p.cta_end = P->n_ctas;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = umma_config(P->n_ctas, P->S, g.smem, st, attr);
    void* args[] = {&a};
    CSB_CUDA(cudaLaunchKernelExC(&cfg, pick_umma(0, NB, P->MT), args));
    return CSB_OK;
}

int launch_umma_pack(const float* X, int64_t ldx, int nb, int cols, int NB, uint8_t* xp, cudaStream_t st) {
    const int vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0 && ldx % 4 == 0;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 1;
    const int windows = (cols + kUmmaWindow - 1) / kUmmaWindow;
    cfg.gridDim = dim3((unsigned)windows); cfg.blockDim = dim3((unsigned)NB * 8);
    CSB_CUDA(cudaLaunchKernelEx(&cfg, NB == 16 ? csb_umma_pack_kernel<16> : NB == 32 ? csb_umma_pack_kernel<32> : csb_umma_pack_kernel<64>, X, (long long)ldx, nb,
                                cols, vec, xp, bad_words(xp, windows)));
    return CSB_OK;
}

// Packs fp32 inputs into xp (umma_xp_bytes) and launches, 64 batch columns at a time.
int launch_umma_fp32(const csb_matrix* A, const UmmaPlan* P, uint8_t* xp, const float* X, int64_t ldx, int batch, float* Y, int64_t ldy, cudaStream_t st) {
    for (int b0 = 0; b0 < batch; b0 += 64) {
        const int nb = std::min(64, batch - b0), NB = umma_nb(nb);
        int rc = launch_umma_pack(X + (int64_t)b0 * ldx, ldx, nb, (int)A->cols, NB, xp, st);
        if (rc == CSB_OK) rc = launch_umma_packed(A, P, xp, Y + (int64_t)b0 * ldy, NB, nb, ldy, st);
        if (rc != CSB_OK) return rc;
    }
    return CSB_OK;
}

// Returns CSB_OK after launching, or 1 when the path does not take the matrix.
int launch_umma(const csb_matrix* A, UmmaPlan* P, const float* X, int64_t ldx, int batch, float* Y, int64_t ldy, void* stream) {
    const int rc = make_umma_plan(A, P);
    return rc != CSB_OK ? rc : launch_umma_fp32(A, P, P->d_xp, X, ldx, batch, Y, ldy, (cudaStream_t)stream);
}

}  // namespace csb
