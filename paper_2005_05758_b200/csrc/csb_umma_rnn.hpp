// The batched recurrent stacks on tcgen05: what csb_umma.cu, csb_umma_upload.cpp, csb_umma_rnn.cu and csb_rnn_step.cu share.
#pragma once

#include <cuda_runtime.h>

#include <memory>

#include "csb_umma.hpp"

namespace csb {

// csb_umma.cu
int umma_clusters(const csb_matrix* A, int (&n)[kUmmaMaxS + 1]);
const void* pick_umma(int mode, int NB, int MT);
struct UmmaStages { int x_depth, w_bytes; size_t smem; };
bool umma_stages(int mode, int NB, int MT, int max_round, size_t room, UmmaStages* out);
int launch_umma_fp32(const csb_matrix* A, const UmmaPlan* P, uint8_t* xp, const float* X, int64_t ldx, int batch, float* Y, int64_t ldy, cudaStream_t st);

// csb_umma_upload.cpp
int upload_umma(const csb_matrix* A, int n, const UmmaHostPlan* H, bool with_xp, UmmaPlan* P);
int make_umma_plan(const csb_matrix* A, UmmaPlan* P);   // 1: the path does not take the matrix

// The layouts of a stack's layers, for every batch size.
struct UmmaStack {
    std::vector<uint64_t> uids;
    int gates = 0, L = 0, H = 0, device = -1;
    int in_size[kMaxLayers] = {};
    bool refused = false;              // a layer does not suit the layout
    bool resident = false;             // one grid holds all layers: the time loop serves it
    bool laid_out = false;             // only then are there plans
    int clusters[kUmmaMaxS + 1] = {};
    int MT = 1, S = 1, flush = 1;      // shape of a resident stack
    int max_round = 0;
    UmmaPlan plan[kMaxLayers];
    ~UmmaStack();
};
// csb_umma_rnn.cu.  for_loop: for the time loop, so that a stack that one grid does not hold is not laid out; *out null: not taken
int umma_stack(int gates, int L, const csb_matrix* const* W, const int* in_size, int H, bool for_loop, std::shared_ptr<UmmaStack>* out);

}  // namespace csb
