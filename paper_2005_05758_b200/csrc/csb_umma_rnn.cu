// LSTM and GRU stacks at larger batch as one launch per sequence on tcgen05 tensor cores: host side of the time loop of
// csb_umma_kernel.cuh, and the layouts of the layers, which the step-by-step form (csb_rnn_step.cu) shares.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <list>
#include <memory>
#include <mutex>
#include <vector>

#include "csb_host.hpp"
#include "csb_rnn1.hpp"
#include "csb_umma_rnn.hpp"
#include "csb_umma_kernel.cuh"

namespace csb {

#define CSB_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            set_error("%s failed: %s", #call, cudaGetErrorString(e_));                     \
            return e_ == cudaErrorMemoryAllocation ? CSB_ERR_ALLOC : CSB_ERR_CUDA;         \
        }                                                                                  \
    } while (0)

UmmaStack::~UmmaStack() { for (UmmaPlan& p : plan) drop_umma_plan(p); }

// What a call of one batch size writes.
struct UmmaRnnPlan {
    std::shared_ptr<UmmaStack> stack;
    int B = 0, NB = 0;
    uint8_t* d_xp[kMaxLayers] = {};    // two buffers of operand images per layer, and 16 bytes of marks for each
    float* d_state = nullptr;          // [L, B, H] c (LSTM) or h (GRU) at the start
    float* d_ends = nullptr;           // [4][L, B, H] h0 and c0 from the host; hT and cT where the caller's arrays cannot be written directly
    uint32_t* d_count = nullptr;
    uint32_t calls = 0;                // counted, so that a mark of an earlier call is told from this one's
    uint32_t* h_status = nullptr; uint32_t* d_status = nullptr;
    float* d_stage = nullptr;          // host-I/O staging of x and y
    size_t stage_cap = 0;
    uint8_t* d_all = nullptr;          // the allocation that all of them but the staging lie in
    ~UmmaRnnPlan() {
        cudaFree(d_all); cudaFree(d_stage);
        if (h_status) cudaFreeHost(h_status);
    }
};

static std::mutex g_umma_mu;
static std::list<std::shared_ptr<UmmaStack>> g_stacks;
static std::list<std::unique_ptr<UmmaRnnPlan>> g_umma_plans;

void drop_umma_rnn_plans(const csb_matrix* A) {
    std::lock_guard<std::mutex> lk(g_umma_mu);
    int prev = 0;
    cudaGetDevice(&prev);
    auto uses = [&](const UmmaStack& s) { return std::find(s.uids.begin(), s.uids.end(), A->uid) != s.uids.end(); };
    for (auto it = g_umma_plans.begin(); it != g_umma_plans.end();) {
        if (uses(*(*it)->stack)) { cudaSetDevice((*it)->stack->device); it = g_umma_plans.erase(it); }
        else ++it;
    }
    for (auto it = g_stacks.begin(); it != g_stacks.end();) {
        if (uses(**it)) { cudaSetDevice((*it)->device); it = g_stacks.erase(it); }
        else ++it;
    }
    cudaSetDevice(prev);
}

static int stack_windows(const UmmaStack& K, int l) { return (K.in_size[l] + K.H + kUmmaWindow - 1) / kUmmaWindow; }

// Does one grid hold the stack, and in which shape?  1 when the device takes none.
static int shape_stack(const csb_matrix* const* W, UmmaStack* K) {
    int* clusters = K->clusters;
    const int rc = umma_clusters(W[0], K->clusters);
    if (rc != CSB_OK) return rc;
    if (clusters[1] < 1) return 1;
    const int tiles = (K->H + 31) / 32;
    int most = 0, least = 0x7fffffff;
    int64_t blocks = 0x7fffffff;
    for (int l = 0; l < K->L; ++l) { most = std::max(most, stack_windows(*K, l)); least = std::min(least, stack_windows(*K, l)); blocks = std::min(blocks, W[l]->nblk); }
    // One grid for all layers, every CTA there for the whole sequence: the shape whose slowest layer costs least (as in
    // umma_shape, with a step's cluster and counter on top whatever the shape).
    double best = 1e300;
    for (int mt = kUmmaMaxMT; mt >= 1; --mt)
        for (int s = 1; s <= std::min<int>(kUmmaMaxS, least); ++s) {
            if (K->L * ((tiles + mt - 1) / mt) > clusters[s]) continue;
            const double cost = umma_cost(mt, s, most);
            if (cost < best) { best = cost; K->MT = mt; K->S = s; }
        }
    K->resident = best < 1e300;
    K->flush = umma_flush(most, blocks);
    return CSB_OK;
}

// The layouts of the layers; 1 when the layout does not take one.
static int lay_out_stack(const csb_matrix* const* W, UmmaStack* K) {
    const int tiles = (K->H + 31) / 32;
    std::vector<UmmaHostPlan> H((size_t)K->L);
    std::atomic<int> next{0};
    std::atomic<bool> failed{false};
    run_on_threads(K->L, [&]() {                           // the layers side by side
        for (int l; (l = next.fetch_add(1)) < K->L && !failed;) {
            try {
                UmmaHostPlan& h = H[(size_t)l];
                h.windows = stack_windows(*K, l);
                h.seg_words = umma_seg_words(W[l]->block_c);
                h.flush = K->flush;
                h.threads = std::max(1, 16 / K->L);
                if (K->resident) { h.MT = K->MT; h.S = K->S; }
                else umma_shape(tiles, h.windows, K->clusters, &h.MT, &h.S);
                h.quads = umma_gate_quads(K->gates, K->in_size[l], K->H, h.MT);
                h.n_groups = (int)(h.quads.size() / (size_t)(4 * h.MT));
                plan_umma_host(W[l], &h);
            } catch (const std::bad_alloc&) { failed = true; }
        }
    });
    if (failed) return CSB_ERR_ALLOC;
    const int rc = upload_umma(W[0], K->L, H.data(), false, K->plan);
    if (rc != CSB_OK) { cudaGetLastError(); return rc; }
    for (int l = 0; l < K->L; ++l) K->max_round = std::max(K->max_round, K->plan[l].max_round);
    UmmaStages g;
    if (K->resident)
        for (int NB = 16; NB <= 32; NB *= 2) {
            if (!umma_stages(1, NB, K->MT, K->max_round, W[0]->smem_optin, &g)) { K->resident = false; break; }
            CSB_CUDA(cudaFuncSetAttribute(pick_umma(K->gates == 4 ? 1 : 2, NB, K->MT), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W[0]->smem_optin));
        }
    return CSB_OK;
}

int umma_stack(int gates, int L, const csb_matrix* const* W, const int* in_size, int H, bool for_loop, std::shared_ptr<UmmaStack>* out) {
    out->reset();
    for (int l = 0; l < L; ++l) if (!umma_applicable(W[l]) || W[l]->nnz == 0) return CSB_OK;
    std::lock_guard<std::mutex> lk(g_umma_mu);
    std::shared_ptr<UmmaStack> K;
    for (auto& s : g_stacks) {
        bool same = s->gates == gates && s->L == L && s->H == H;
        for (int l = 0; l < L && same; ++l) same = s->uids[l] == W[l]->uid;
        if (same) { K = s; break; }
    }
    if (!K) {
        K = std::make_shared<UmmaStack>();
        K->gates = gates; K->L = L; K->H = H; K->device = W[0]->device;
        for (int l = 0; l < L; ++l) { K->uids.push_back(W[l]->uid); K->in_size[l] = in_size[l]; }
        const int rc = shape_stack(W, K.get());
        if (rc != CSB_OK && rc != 1) return rc;
        K->refused = rc == 1;
        g_stacks.push_back(K);
    }
    if (K->refused || (for_loop && !K->resident)) return CSB_OK;
    if (!K->laid_out) {
        const int rc = guarded([&] { return lay_out_stack(W, K.get()); });
        K->laid_out = rc == CSB_OK && (K->resident || !for_loop);
        if (!K->laid_out) for (UmmaPlan& p : K->plan) drop_umma_plan(p);
        if (rc != CSB_OK && rc != 1 && rc != CSB_ERR_ALLOC) return rc;
        // (where memory does not reach for these layouts, those of the step-by-step form may still fit; for good, so that a
        // stack keeps its bits)
        K->refused = rc != CSB_OK;
    }
    if (K->laid_out) *out = K;
    return CSB_OK;
}

// What a sequence starts from: x_0 and h0 as operand images, the cells' states, the counter.
struct UmmaBeginArgs {
    const float* x; const float* h0; const float* c0;     // h0, c0: null = zeros
    float* state; uint32_t* count;
    uint8_t* xp[kMaxLayers];
    uint32_t* bad[kMaxLayers];
    int in_size[kMaxLayers], windows[kMaxLayers];
    int L, B, H, lstm, x_vec;
    uint32_t call;
};
template <int NB>
__global__ void __launch_bounds__(256) csb_umma_begin_kernel(const __grid_constant__ UmmaBeginArgs a) {
    const int chunks = (a.in_size[0] + 7) / 8, n = a.L * a.B * a.H;
    const long long all = (long long)n + (long long)chunks * a.B;
    auto mark = [&](int l) { *reinterpret_cast<uint2*>(a.bad[l] + 4 * (l & 1)) = make_uint2(a.call, (uint32_t)l + 1u); };
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.count = 0u;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < all; i += (long long)gridDim.x * blockDim.x) {
        if (i < n) {
            const int u = (int)(i % a.H), b = (int)(i / a.H % a.B), l = (int)(i / a.H / a.B);
            const float h = a.h0 ? a.h0[i] : 0.f;
            // (layer l reads its first step in tick l)
            if (put_value<NB>(a.xp[l] + (size_t)(l & 1) * a.windows[l] * (NB * 256), b, a.in_size[l] + u, h)) mark(l);
            a.state[i] = !a.lstm ? h : a.c0 ? a.c0[i] : 0.f;
        } else {
            const int j = (int)(i - n), b = j / chunks, c = (j - b * chunks) * 8;
            if (put_eight<NB>(a.xp[0], b, c, a.in_size[0], a.x + (size_t)b * a.in_size[0] + c, a.x_vec != 0)) mark(0);
        }
    }
}

static int build_plan(UmmaRnnPlan* P) {
    const UmmaStack& K = *P->stack;
    const size_t ns = (size_t)K.L * P->B * K.H * 4;
    size_t bytes = 0, xp[kMaxLayers];
    auto room = [&bytes](size_t more) { const size_t here = bytes; bytes += (more + 255) / 256 * 256; return here; };
    for (int l = 0; l < K.L; ++l) xp[l] = room((size_t)2 * K.plan[l].windows * P->NB * 256 + 32);
    const size_t images = bytes, state = room(ns), ends = room(4 * ns), count = room(4);
    CSB_CUDA(cudaMalloc((void**)&P->d_all, bytes));
    // what is not written (columns past the last, batch columns past B) stays zero
    CSB_CUDA(cudaMemsetAsync(P->d_all, 0, images, cudaStreamPerThread));
    for (int l = 0; l < K.L; ++l) P->d_xp[l] = P->d_all + xp[l];
    P->d_state = reinterpret_cast<float*>(P->d_all + state);
    P->d_ends = reinterpret_cast<float*>(P->d_all + ends);
    P->d_count = reinterpret_cast<uint32_t*>(P->d_all + count);
    CSB_CUDA(cudaHostAlloc((void**)&P->h_status, 4, cudaHostAllocMapped));
    *P->h_status = 0;
    CSB_CUDA(cudaHostGetDevicePointer((void**)&P->d_status, P->h_status, 0));
    CSB_CUDA(cudaStreamSynchronize(cudaStreamPerThread));
    return CSB_OK;
}

int rnn_forward_umma(int gates, int L, const csb_matrix* const* W, const float* const* bias, const float* x, int64_t T, int B, int H, const int* in_size,
                     const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags, void* stream) {
    if (B > 32 || T > 0x3fffffff || (getenv("CSB_RNN_STEP_UNPACKED") && atoi(getenv("CSB_RNN_STEP_UNPACKED")))) return 1;
    std::shared_ptr<UmmaStack> K;
    int rc = umma_stack(gates, L, W, in_size, H, true, &K);
    if (rc != CSB_OK) return rc;
    if (!K) return 1;
    UmmaRnnPlan* P = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_umma_mu);
        for (auto& p : g_umma_plans) if (p->stack == K && p->B == B) P = p.get();
        if (!P) {
            std::unique_ptr<UmmaRnnPlan> np(new UmmaRnnPlan());
            np->stack = K; np->B = B; np->NB = B <= 16 ? 16 : 32;
            if ((rc = build_plan(np.get())) != CSB_OK) { cudaGetLastError(); return rc == CSB_ERR_ALLOC ? 1 : rc; }
            P = np.get();
            g_umma_plans.push_back(std::move(np));
        }
        ++P->calls;
    }
    UmmaStages g;
    if (!umma_stages(1, P->NB, K->plan[0].MT, K->max_round, W[0]->smem_optin, &g)) return 1;
    // (as the step-by-step forms count: rows of their product, two per sequence for the GRU)
    note_tensor_kernel(kTensorLoop);
    note_recurrent_path((gates == 3 ? 2 : 1) * B <= 32 ? kPathStepsPacked : kPathSteps);
    cudaStream_t st = (cudaStream_t)stream;
    const bool host_io = (flags & CSB_FLAG_HOST_IO) != 0, lstm = gates == 4;
    const int NB = P->NB;
    const size_t nx = (size_t)T * B * in_size[0], ny = y ? (size_t)T * B * H : 0, ns = (size_t)L * B * H;
    const float* dx = x;
    float* dy = y;
    if (!lstm) { c0 = nullptr; cT = nullptr; }
    if (host_io) {
        const size_t need = nx + ny;
        if (need > P->stage_cap) {
            CSB_CUDA(cudaStreamSynchronize(st));
            cudaFree(P->d_stage); P->d_stage = nullptr; P->stage_cap = 0;
            CSB_CUDA(cudaMalloc((void**)&P->d_stage, need * 4));
            P->stage_cap = need;
        }
        CSB_CUDA(cudaMemcpyAsync(P->d_stage, x, nx * 4, cudaMemcpyHostToDevice, st));
        dx = P->d_stage;
        dy = y ? P->d_stage + nx : nullptr;
        if (h0) { CSB_CUDA(cudaMemcpyAsync(P->d_ends, h0, ns * 4, cudaMemcpyHostToDevice, st)); h0 = P->d_ends; }
        if (c0) { CSB_CUDA(cudaMemcpyAsync(P->d_ends + ns, c0, ns * 4, cudaMemcpyHostToDevice, st)); c0 = P->d_ends + ns; }
    }
    // The initial states are read by the launch in front of the loop, so final states may lie on them; final states that
    // overlap another output are copied there after it.
    auto meets = [](const float* p, size_t n, const float* q, size_t m) { return p && q && n && m && p < q + m && q < p + n; };
    const bool states_meet = meets(hT, ns, cT, ns);
    const bool move_hT = hT && (host_io || states_meet || meets(hT, ns, y, ny)), move_cT = cT && (host_io || states_meet || meets(cT, ns, y, ny));
    UmmaBeginArgs ba{};
    ba.x = dx; ba.h0 = h0; ba.c0 = c0; ba.state = P->d_state; ba.count = P->d_count; ba.L = L; ba.B = B; ba.H = H; ba.lstm = lstm;
    ba.x_vec = (reinterpret_cast<uintptr_t>(dx) & 15) == 0 && in_size[0] % 4 == 0;
    UmmaArgs a{};
    a.n_parts = L; a.nb = B; a.status = P->d_status; a.S = K->plan[0].S; a.flush = K->plan[0].flush;
    a.x_depth = g.x_depth; a.w_bytes = g.w_bytes;
    int ctas = 0;
    for (int l = 0; l < L; ++l) {
        const UmmaPlan& Q = K->plan[l];
        UmmaPart& p = a.part[l];
        p.stream = Q.d_stream; p.ctas = Q.d_ctas; p.rounds = Q.d_rounds; p.quads = Q.d_quads; p.xp = P->d_xp[l];
        p.bad = ba.bad[l] = reinterpret_cast<uint32_t*>(P->d_xp[l] + (size_t)2 * Q.windows * NB * 256);
        p.block_r = W[l]->block_r; p.seg_words = Q.seg_words; p.windows = Q.windows;
        ctas += Q.n_ctas;
        p.cta_end = ctas;
        a.bias[l] = bias ? bias[l] : nullptr;
        a.in_size[l] = in_size[l];
        ba.xp[l] = P->d_xp[l]; ba.in_size[l] = in_size[l]; ba.windows[l] = Q.windows;
    }
    a.x = dx; a.y = dy; a.state0 = P->d_state;
    a.hT = move_hT ? P->d_ends + 2 * ns : hT;
    a.cT = move_cT ? P->d_ends + 3 * ns : cT;
    a.count = P->d_count; a.T = (int)T; a.H = H; a.x_vec = ba.x_vec; a.call = ba.call = P->calls;
    uint32_t extra = 0;
    barrier_test_hook(&extra, &a.limit_ns);
    a.never = extra == 1 ? kNever : 0u;
    a.never_step = (int)extra - 2;
    *P->h_status = 0;
    const size_t all = ns + (size_t)B * ((in_size[0] + 7) / 8);
    const unsigned blocks = (unsigned)std::min<size_t>((all + 255) / 256, 4096);
    (NB == 16 ? csb_umma_begin_kernel<16> : csb_umma_begin_kernel<32>)<<<blocks, 256, 0, st>>>(ba);
    CSB_CUDA(cudaGetLastError());
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.S; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3(kUmmaThreads); cfg.dynamicSmemBytes = g.smem;
    cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = a.S > 1 ? 2 : 1;
    void* params[] = {&a};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, pick_umma(lstm ? 1 : 2, NB, K->plan[0].MT), params);
    if (e == cudaErrorCooperativeLaunchTooLarge) { cudaGetLastError(); return 1; }     // a device that others share; nothing of the caller's has been written
    CSB_CUDA(e);
    const cudaMemcpyKind kind = host_io ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    if (host_io && y) CSB_CUDA(cudaMemcpyAsync(y, dy, ny * 4, kind, st));
    if (move_hT) CSB_CUDA(cudaMemcpyAsync(hT, a.hT, ns * 4, kind, st));
    if (move_cT) CSB_CUDA(cudaMemcpyAsync(cT, a.cT, ns * 4, kind, st));
    if (host_io || !(flags & CSB_FLAG_ASYNC)) {
        CSB_CUDA(cudaStreamSynchronize(st));
        if (*P->h_status != 0) {
            set_error("the batched time loop gave up a bounded wait (code %u: %s)", *P->h_status,
                      *P->h_status == kDevBarrierTimeout ? "other CTAs" : "a copy or a product");
            return CSB_ERR_TIMEOUT;
        }
    }
    return CSB_OK;
}

}  // namespace csb
