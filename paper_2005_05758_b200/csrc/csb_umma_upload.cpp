// Device side of the plans of the batched product on tcgen05 tensor cores (layout: csb_umma.hpp): allocation and upload.
#include <algorithm>
#include <cstdlib>
#include <new>
#include <vector>

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
    cudaFree(P.d_all);
    P.d_all = nullptr; P.d_stream = nullptr; P.d_ctas = nullptr; P.d_quads = nullptr; P.d_rounds = nullptr; P.d_xp = nullptr;
}

// Uploads n host plans (the layers of a stack; with_xp: and makes room for the packed inputs of a bare product), all in one
// allocation that the first one owns: past 2 MB each allocation takes 0.3 ms, which is what four layers of 3.4 MB spent
// most of their first call on.  1: a round of values does not fit in shared memory.  What is allocated when it fails is
// the caller's to drop.
int upload_umma(const csb_matrix* A, int n, const UmmaHostPlan* H, bool with_xp, UmmaPlan* P) {
    UmmaStages st;
    std::vector<size_t> at((size_t)n * 3);                 // of a plan: values, tables, packed inputs
    size_t bytes = 0;
    auto room = [&bytes](size_t more) { const size_t here = bytes; bytes += (more + 255) / 256 * 256; return here; };
    auto table_bytes = [](const UmmaHostPlan& h) { return h.ctas.size() * sizeof(UmmaCta) + h.quads.size() * sizeof(UmmaQuad) + h.rounds.size() * sizeof(UmmaRound); };
    for (int i = 0; i < n; ++i) {
        P[i].MT = H[i].MT; P[i].S = H[i].S; P[i].n_ctas = (int)H[i].ctas.size(); P[i].windows = H[i].windows; P[i].seg_words = H[i].seg_words;
        P[i].flush = H[i].flush; P[i].max_round = (int)H[i].max_round;
        for (int NB = 16; NB <= 64; NB *= 2) {
            if (!umma_stages(0, NB, H[i].MT, P[i].max_round, A->smem_optin, &st)) return 1;
            CSB_CUDA(cudaFuncSetAttribute(pick_umma(0, NB, H[i].MT), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A->smem_optin));
        }
        at[(size_t)i * 3] = room(H[i].total128 * 128);
        at[(size_t)i * 3 + 1] = room(table_bytes(H[i]));
        at[(size_t)i * 3 + 2] = room(with_xp ? umma_xp_bytes(H[i].windows) : 0);
    }
    CSB_CUDA(cudaMalloc((void**)&P[0].d_all, bytes));
    for (int i = 0; i < n; ++i) {
        UmmaPlan& p = P[i];
        const UmmaHostPlan& h = H[i];
        p.d_stream = P[0].d_all + at[(size_t)i * 3];
        p.d_ctas = reinterpret_cast<UmmaCta*>(P[0].d_all + at[(size_t)i * 3 + 1]);
        p.d_quads = reinterpret_cast<UmmaQuad*>(p.d_ctas + h.ctas.size());
        p.d_rounds = reinterpret_cast<UmmaRound*>(p.d_quads + h.quads.size());
        if (with_xp) p.d_xp = P[0].d_all + at[(size_t)i * 3 + 2];
        for (size_t c = 0; c < h.ctas.size(); ++c)
            if (!h.streams[c].empty())
                CSB_CUDA(cudaMemcpyAsync(p.d_stream + (size_t)h.ctas[c].off128 * 128, h.streams[c].data(), h.streams[c].size(), cudaMemcpyHostToDevice, cudaStreamPerThread));
        CSB_CUDA(cudaMemcpyAsync(p.d_ctas, h.ctas.data(), h.ctas.size() * sizeof(UmmaCta), cudaMemcpyHostToDevice, cudaStreamPerThread));
        CSB_CUDA(cudaMemcpyAsync(p.d_quads, h.quads.data(), h.quads.size() * sizeof(UmmaQuad), cudaMemcpyHostToDevice, cudaStreamPerThread));
        CSB_CUDA(cudaMemcpyAsync(p.d_rounds, h.rounds.data(), h.rounds.size() * sizeof(UmmaRound), cudaMemcpyHostToDevice, cudaStreamPerThread));
    }
    CSB_CUDA(cudaStreamSynchronize(cudaStreamPerThread));
    return CSB_OK;
}

// Out of memory is answered like a matrix that does not suit the layout, by the other form
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
            H.flush = umma_flush(H.windows, A->nblk);
            H.quads = umma_row_quads(A, H.MT);
            H.n_groups = (int)(H.quads.size() / (size_t)(4 * H.MT));
            plan_umma_host(A, &H);
            return upload_umma(A, 1, &H, true, P);
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
