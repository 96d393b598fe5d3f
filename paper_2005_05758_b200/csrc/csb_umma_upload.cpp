// Device side of the plans of the batched product on tcgen05 tensor cores (layout: csb_umma.hpp): allocation and upload.
#include <algorithm>
#include <cstdlib>
#include <new>

#include "csb_umma_rnn.hpp"

namespace csb {

#define CSB_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            set_error("%s failed: %s", #call, cudaGetErrorString(e_));                     \
            return e_ == cudaErrorMemoryAllocation ? CSB_ERR_ALLOC : CSB_ERR_CUDA;         \
        }                                                                                  \
    } while (0)

void drop_umma_plan(UmmaPlan& P) {
    cudaFree(P.d_stream); cudaFree(P.d_ctas); cudaFree(P.d_quads); cudaFree(P.d_rounds); cudaFree(P.d_xp);
    P.d_stream = nullptr; P.d_ctas = nullptr; P.d_quads = nullptr; P.d_rounds = nullptr; P.d_xp = nullptr;
}

// Uploads a host plan; 1: a round of its values does not fit in shared memory.  What is allocated when it fails is the
// caller's to drop.
int upload_umma(const csb_matrix* A, const UmmaHostPlan& H, UmmaPlan* P) {
    P->MT = H.MT; P->S = H.S; P->n_ctas = (int)H.ctas.size(); P->windows = H.windows; P->seg_words = H.seg_words; P->flush = H.flush;
    P->max_round = (int)H.max_round;
    UmmaStages st;
    for (int NB = 16; NB <= 64; NB *= 2) {
        if (!umma_stages(0, NB, H.MT, P->max_round, A->smem_optin, &st)) return 1;
        CSB_CUDA(cudaFuncSetAttribute(pick_umma(0, NB, H.MT), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A->smem_optin));
    }
    CSB_CUDA(cudaMalloc((void**)&P->d_stream, std::max<size_t>(H.total128, 1) * 128));
    for (size_t i = 0; i < H.ctas.size(); ++i)
        if (!H.streams[i].empty())
            CSB_CUDA(cudaMemcpyAsync(P->d_stream + (size_t)H.ctas[i].off128 * 128, H.streams[i].data(), H.streams[i].size(), cudaMemcpyHostToDevice, cudaStreamPerThread));
    CSB_CUDA(cudaMalloc((void**)&P->d_ctas, H.ctas.size() * sizeof(UmmaCta)));
    CSB_CUDA(cudaMemcpyAsync(P->d_ctas, H.ctas.data(), H.ctas.size() * sizeof(UmmaCta), cudaMemcpyHostToDevice, cudaStreamPerThread));
    CSB_CUDA(cudaMalloc((void**)&P->d_quads, H.quads.size() * sizeof(UmmaQuad)));
    CSB_CUDA(cudaMemcpyAsync(P->d_quads, H.quads.data(), H.quads.size() * sizeof(UmmaQuad), cudaMemcpyHostToDevice, cudaStreamPerThread));
    CSB_CUDA(cudaMalloc((void**)&P->d_rounds, H.rounds.size() * sizeof(UmmaRound)));
    CSB_CUDA(cudaMemcpyAsync(P->d_rounds, H.rounds.data(), H.rounds.size() * sizeof(UmmaRound), cudaMemcpyHostToDevice, cudaStreamPerThread));
    CSB_CUDA(cudaStreamSynchronize(cudaStreamPerThread));
    return CSB_OK;
}

// All of a plan's arrays or none.  Out of memory is answered like a matrix that does not suit the layout, by the other form
// (whose layout is a half to a fifth of this one), now and in later calls: a handle keeps its bits.
int make_umma_plan(const csb_matrix* A, UmmaPlan* P) {
    if (P->built || P->unusable) return P->built ? CSB_OK : 1;
    const int rc = [&]() -> int {
        try {
            UmmaHostPlan H;
            H.windows = (int)((A->cols + kUmmaWindow - 1) / kUmmaWindow);
            H.seg_words = umma_seg_words(A->block_c);
            int clusters[kUmmaMaxS + 1];
            const int crc = umma_clusters(A, clusters);
            if (crc != CSB_OK) return crc;
            if (clusters[1] < 1) return 1;
            umma_shape((int)((A->rows + 127) / 128), H.windows, clusters, &H.MT, &H.S);
            H.flush = umma_flush(H.windows);
            H.quads = umma_row_quads(A, H.MT);
            H.n_groups = (int)(H.quads.size() / (size_t)(4 * H.MT));
            plan_umma_host(A, &H);
            CSB_CUDA(cudaMalloc((void**)&P->d_xp, umma_xp_bytes(H.windows)));
            return upload_umma(A, H, P);
        } catch (const std::bad_alloc&) { return CSB_ERR_ALLOC; }
    }();
    if (rc == CSB_OK) { P->built = true; return CSB_OK; }
    drop_umma_plan(*P);
    cudaGetLastError();
    if (rc != 1 && rc != CSB_ERR_ALLOC) return rc;
    P->unusable = true;
    clear_error();
    return 1;
}

bool umma_applicable(const csb_matrix* A) {
    if (getenv("CSB_NO_UMMA") && atoi(getenv("CSB_NO_UMMA"))) return false;
    return A->val_dtype == CSB_F16 && A->device >= 0 && umma_seg_words(A->block_c) > 0;
}

}  // namespace csb
