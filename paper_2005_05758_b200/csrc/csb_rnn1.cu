// Launch glue of the resident time loop (kernel: csb_rnn1_kernel.cuh).
#include <cstdlib>
#include <list>
#include <memory>
#include <mutex>

#include "csb_rnn1_args.hpp"
#include "csb_device.cuh"

namespace csb {

#define CSB_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            set_error("%s failed: %s", #call, cudaGetErrorString(e_));                     \
            return e_ == cudaErrorMemoryAllocation ? CSB_ERR_ALLOC : CSB_ERR_CUDA;         \
        }                                                                                  \
    } while (0)

#ifdef CSB_PHASE_CLOCKS
static long long* g_r1_clocks = nullptr;
static int g_r1_clock_ctas = 0;
extern "C" int csb_debug_rnn1_clocks(long long* host_out, int max_ctas) {
    cudaMemcpy(host_out, g_r1_clocks, (size_t)std::min(max_ctas, g_r1_clock_ctas) * 8 * 8, cudaMemcpyDeviceToHost);
    return g_r1_clock_ctas;
}
#endif

// Device memory that goes together.
struct R1Memory {
    std::vector<void*> p;
    ~R1Memory() { for (void* q : p) cudaFree(q); }
};
// Everything one (cell, layer stack, batch size) needs on the device; built on first use and kept until one of
// its matrices is freed.  The weights' layout is shared by the batch sizes of a tile; what a call writes is not, since calls
// of different batch sizes may overlap.
struct Rnn1Plan {
    int cell = 0, L = 0, B = 0, BT = 1, device = 0, n_ctas = 0, H = 0, S = 0, val_dtype = 0;
    bool unusable = false;
    std::vector<uint64_t> uids;
    bool unit_loop = false;                    // csb_rnn_unit_kernel.cuh, else csb_rnn1_kernel.cuh
    R1Args a{};
    RuArgs u{};
    size_t smem = 0;
    const void* kernel = nullptr;
    std::shared_ptr<R1Memory> layout = std::make_shared<R1Memory>();
    R1Memory own;
    uint32_t* h_status = nullptr;
    float* d_stage = nullptr; size_t stage_cap = 0;      // x and y of calls with host arrays
    float* d_x = nullptr; size_t x_cap = 0;              // x of calls that write over it
    float* d_states = nullptr;                 // [h0, c0, hT, cT] of calls with host arrays or with states in each other's places
    ~Rnn1Plan() {
        cudaFree(d_stage);
        if (h_status) cudaFreeHost(h_status);
    }
};
static std::mutex g_r1_mu;
static std::list<std::unique_ptr<Rnn1Plan>> g_r1_plans;

void drop_rnn1_plans(const csb_matrix* A) {
    std::lock_guard<std::mutex> lk(g_r1_mu);
    int prev = 0;
    cudaGetDevice(&prev);
    for (auto it = g_r1_plans.begin(); it != g_r1_plans.end();) {
        if (std::find((*it)->uids.begin(), (*it)->uids.end(), A->uid) != (*it)->uids.end()) {
            cudaSetDevice((*it)->device);
            it = g_r1_plans.erase(it);
        } else ++it;
    }
    cudaSetDevice(prev);
}

static const void* pick_kernel_bt(int cell, int BT, int val_dtype) {
    return BT == 1 ? r1_kernel_b1(cell, val_dtype) : BT == 4 ? r1_kernel_b4(cell, val_dtype) : r1_kernel_b8(cell, val_dtype);
}

static int env_int(const char* name, int dflt) {
    const char* v = getenv(name);
    return v && *v ? atoi(v) : dflt;
}

template <typename V>
static int put(R1Memory* M, const std::vector<V>& h, V** d) {
    CSB_CUDA(cudaMalloc((void**)d, std::max<size_t>(h.size(), 1) * sizeof(V)));
    M->p.push_back(*d);
    if (!h.empty()) CSB_CUDA(cudaMemcpy(*d, h.data(), h.size() * sizeof(V), cudaMemcpyHostToDevice));
    return CSB_OK;
}

// What a call writes: exchange buffers, step numbers and progress (all from zero), states, the status word.
static int build_state(Rnn1Plan* P) {
    R1Common& c = P->unit_loop ? (R1Common&)P->u : (R1Common&)P->a;
    size_t bytes = 0;
    auto room = [&](size_t n) { const size_t at = bytes; bytes += (n + 255) & ~(size_t)255; return at; };
    size_t ex[2][kMaxLayers] = {};
    for (int e = 0; e < r1_ops(P->cell); ++e)
        for (int l = 0; l < P->L; ++l) {
            const size_t pairs = ((size_t)(e ? P->H : P->S) * P->BT + 1) & ~(size_t)1;
            ex[e][l] = room(kR1Ring * (P->unit_loop ? pairs * sizeof(uint2) : (size_t)P->a.words[e][l] * sizeof(uint4)));
        }
    const size_t epoch = room((size_t)P->n_ctas * 4), progress = room((size_t)kMaxLayers * 4), states = room((size_t)2 * P->L * P->B * (P->S + P->H) * 4);
    uint8_t* d = nullptr;
    CSB_CUDA(cudaMalloc((void**)&d, bytes));
    P->own.p.push_back(d);
    CSB_CUDA(cudaMemset(d, 0, bytes));
    for (int e = 0; e < r1_ops(P->cell); ++e)
        for (int l = 0; l < P->L; ++l) {
            if (P->unit_loop) P->u.ex[e][l] = reinterpret_cast<uint2*>(d + ex[e][l]);
            else P->a.ex[e][l] = reinterpret_cast<uint4*>(d + ex[e][l]);
        }
    c.epoch = reinterpret_cast<uint32_t*>(d + epoch); c.progress = reinterpret_cast<uint32_t*>(d + progress);
    P->d_states = reinterpret_cast<float*>(d + states);
    CSB_CUDA(cudaHostAlloc((void**)&P->h_status, 4, cudaHostAllocMapped));
    *P->h_status = 0;
    CSB_CUDA(cudaHostGetDevicePointer((void**)&c.status, P->h_status, 0));
    CSB_CUDA(cudaDeviceSynchronize());
    return CSB_OK;
}
// Whether the grid can be resident at once.
static int fits(Rnn1Plan* P, const csb_matrix* A0, bool* yes) {
    *yes = false;
    if (P->smem > A0->smem_optin) return CSB_OK;
    CSB_CUDA(cudaFuncSetAttribute(P->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A0->smem_optin));
    int occ = 0;
    CSB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, P->kernel, kR1Threads, P->smem));
    *yes = occ >= 1 && P->n_ctas <= occ * A0->sm_count;
    return CSB_OK;
}

static void fill_common(R1Common& c, int L, const int* in_size, const int* layer_ctas, int H, int S) {
    for (int l = 0; l < L; ++l) { c.in_size[l] = in_size[l]; c.layer_ctas[l] = layer_ctas[l]; }
    c.H = H; c.S = S; c.L = L;
}

// The unit loop's plan; 1 when it is not the one for these matrices.
static int build_unit_plan(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, int64_t weights,
                           Rnn1Plan* P) {
    if (env_int("CSB_RNN_NO_UNIT", 0)) return 1;           // diagnostics: the other loop, which covers every size of this one
    const csb_matrix* A0 = W[0];
    int max_in = 0;
    for (int l = 0; l < L; ++l) max_in = std::max(max_in, in_size[l]);
    // Taken wherever its lists fit in shared memory: 4 (fp16) or 8 bytes a weight, uneven CTAs and padding one part in
    // eight (an estimate that spares the planning; fits() decides).  Below that line it was the faster loop at every
    // size measured except one, level there: 1024 units and 16 k weights a CTA 1.9 against 3.7 us a step, LSTMP
    // 3.0 / 5.9, 8 batch columns 4.2 / 5.9, 2 x 1024 units on 1024 inputs 3.2 / 3.0, 2048 units on 2048 3.2 / 3.3.
    const size_t lists = (size_t)weights * (W[0]->val_dtype == CSB_F16 ? 4 : 8) / (size_t)A0->sm_count * 9 / 8;
    if (lists + (size_t)(2 * (max_in + S) + H) * BT * 4 > A0->smem_optin) return 1;
    // A unit per warp where a step is a chain of latencies (batch 1: more CTAs make the exchange longer, 2.6 us with 8
    // units a CTA), as many CTAs as there are where batch columns make it the product's time (4.3 against 6.1 us).
    const int64_t units = (int64_t)L * H, each = BT == 1 ? kR1Warps : kR1Warps / 4;
    int want = (int)std::min<int64_t>(A0->sm_count, std::max<int64_t>(L, (units + each - 1) / each));
    want = std::min(A0->sm_count, env_int("CSB_R1_CTAS", want));
    RuHostPlan Hp;
    const int hrc = plan_unit_host(cell, L, W, Wp, in_size, H, S, BT, want, &Hp);
    if (hrc != CSB_OK) return hrc;
    RuArgs& a = P->u;
    size_t at = Hp.max_bytes;
    auto room = [&](size_t floats) { const size_t o = at; at = (at + floats * 4 + 15) & ~(size_t)15; return (uint32_t)o; };
    const int ops = r1_ops(cell);
    for (uint32_t& v : a.vu) v = room((size_t)(max_in + 1) * BT);
    for (uint32_t& v : a.vr) v = room((size_t)(S + 1) * BT);
    a.vm = room(ops == 2 ? (size_t)(H + 1) * BT : 0);
    a.misc = room(4);
    P->smem = at;
    P->n_ctas = (int)Hp.ctas.size();
    P->kernel = BT == 1 ? ru_kernel_b1(cell, P->val_dtype) : BT == 4 ? ru_kernel_b4(cell, P->val_dtype) : ru_kernel_b8(cell, P->val_dtype);
    bool yes = false;
    int rc = fits(P, A0, &yes);
    if (rc != CSB_OK) return rc;
    if (!yes) return 1;
    uint8_t* d_img = nullptr; RuCta* d_ctas = nullptr;
    if ((rc = put(P->layout.get(), Hp.bytes, &d_img)) != CSB_OK || (rc = put(P->layout.get(), Hp.ctas, &d_ctas)) != CSB_OK) return rc;
    a.images = d_img; a.ctas = d_ctas;
    fill_common(a, L, in_size, Hp.layer_ctas, H, S);
    P->unit_loop = true;
    return CSB_OK;
}

// Layout of the weights, uploaded.  Returns 1 (and marks the plan) when neither kernel takes these matrices.
static int build_layout(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, Rnn1Plan* P) {
    const csb_matrix* A0 = W[0];
    P->cell = cell; P->L = L; P->BT = BT; P->device = A0->device; P->H = H; P->S = S; P->val_dtype = A0->val_dtype;
    P->unusable = true;
    for (int l = 0; l < L; ++l) P->uids.push_back(W[l]->uid);
    if (Wp) for (int l = 0; l < L; ++l) P->uids.push_back(Wp[l]->uid);
    int64_t weights = 0;
    for (int l = 0; l < L; ++l) {
        weights += W[l]->nnz + (Wp ? Wp[l]->nnz : 0);
        if (W[l]->val_dtype != A0->val_dtype || (Wp && Wp[l]->val_dtype != A0->val_dtype)) return 1;
    }
    {
        const int rc = build_unit_plan(cell, L, W, Wp, in_size, H, S, BT, weights, P);
        if (rc == CSB_OK) { P->unusable = false; return CSB_OK; }
        if (rc != 1) return rc;
    }
    if (BT == 8 && P->val_dtype != CSB_F16) return 1;      // not built for fp32 values
    int want = (int)std::min<int64_t>(A0->sm_count, std::max<int64_t>(L, weights / env_int("CSB_R1_MIN", 1024)));
    want = std::min(A0->sm_count, env_int("CSB_R1_CTAS", want));
    R1HostPlan Hp;
    const int hrc = plan_rnn1_host(cell, L, W, Wp, in_size, H, S, BT, want, A0->smem_optin, &Hp);
    if (hrc != CSB_OK) return hrc;
    R1Args& a = P->a;
    int max_in = 0;
    for (int l = 0; l < L; ++l) max_in = std::max(max_in, in_size[l]);
    const R1Carve M(Hp, cell, max_in, H, S, BT);
    for (int i = 0; i < 2; ++i) { a.vu[i] = M.vu[i]; a.part[i] = M.part[i]; a.z[i] = M.z[i]; }
    a.vr = M.vr; a.vm = M.vm; a.cs = M.cs; a.bias0 = M.bias0; a.bias1 = M.bias1; a.misc = M.misc;
    P->smem = M.total;
    P->n_ctas = (int)Hp.ctas.size();
    P->kernel = pick_kernel_bt(cell, BT, P->val_dtype);
    bool yes = false;
    int rc = fits(P, A0, &yes);
    if (rc != CSB_OK) return rc;
    if (!yes) return 1;
    uint8_t* d_img = nullptr; R1Cta* d_ctas = nullptr;
    if ((rc = put(P->layout.get(), Hp.bytes, &d_img)) != CSB_OK || (rc = put(P->layout.get(), Hp.ctas, &d_ctas)) != CSB_OK) return rc;
    a.images = d_img; a.ctas = d_ctas;
    for (int e = 0; e < r1_ops(cell); ++e)
        for (int l = 0; l < L; ++l) {
            const std::vector<uint32_t>& m = Hp.wmap[e][l];
            uint32_t* d_map = nullptr;
            if ((rc = put(P->layout.get(), m, &d_map)) != CSB_OK) return rc;
            a.wmap[e][l] = d_map; a.words[e][l] = (int)m.size();
        }
    fill_common(a, L, in_size, Hp.layer_ctas, H, S);
    P->unusable = false;
    return CSB_OK;
}

int rnn1_forward(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const float* const* bias, const float* x, int64_t T, int B,
                 int H, int S, const int* in_size, const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags, void* stream) {
    if (env_int("CSB_RNN_NO_RNN1", 0)) return 1;
    if (B > 1 && env_int("CSB_RNN_NO_STEPWISE", 0)) return 1;   // asks for the persistent kernel of csb_rnn.cu
    const int BT = B == 1 ? 1 : B <= 4 ? 4 : 8;            // tiles of batch columns that the kernels are built for
    if (B > 8 || T > 0x7fffffff) return 1;                 // (the kernels count steps in 32 bits)
    Rnn1Plan* P = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_r1_mu);
        Rnn1Plan* like = nullptr;                          // a plan of the same tile: its layout serves
        for (auto& p : g_r1_plans) {
            if (p->cell != cell || p->L != L || p->BT != BT) continue;
            bool same = true;
            for (int l = 0; l < L; ++l) same = same && p->uids[l] == W[l]->uid && (!Wp || p->uids[L + l] == Wp[l]->uid);
            if (!same) continue;
            if (p->B == B) { P = p.get(); break; }
            like = p.get();
        }
        if (!P) {
            std::unique_ptr<Rnn1Plan> np(new Rnn1Plan());
            int rc = CSB_OK;
            if (like) {
                np->cell = like->cell; np->L = like->L; np->BT = like->BT; np->device = like->device; np->n_ctas = like->n_ctas; np->H = like->H; np->S = like->S;
                np->val_dtype = like->val_dtype; np->unusable = like->unusable; np->uids = like->uids; np->unit_loop = like->unit_loop;
                np->a = like->a; np->u = like->u; np->smem = like->smem; np->kernel = like->kernel; np->layout = like->layout;
            } else {
                try { rc = build_layout(cell, L, W, Wp, in_size, H, S, BT, np.get()); }
                catch (const std::bad_alloc&) { set_error("out of host memory while planning the time loop"); rc = CSB_ERR_ALLOC; }
            }
            np->B = B;
            if (rc == CSB_OK && !np->unusable) rc = build_state(np.get());
            if (rc != CSB_OK && rc != 1) return rc;
            P = np.get();
            g_r1_plans.push_back(std::move(np));
        }
    }
    if (P->unusable) return 1;
    note_recurrent_path(P->unit_loop ? kPathUnitLoop : kPathBlockLoop);
    cudaStream_t st = (cudaStream_t)stream;
    const bool host_io = (flags & CSB_FLAG_HOST_IO) != 0, has_c = cell == kR1Lstm || cell == kR1Lstmp;
    const size_t nx = (size_t)T * B * in_size[0], ny = y ? (size_t)T * B * S : 0, nh = (size_t)L * B * S, nc = has_c ? (size_t)L * B * H : 0;
    R1Args a1 = P->a;
    RuArgs au = P->u;
    R1Common& a = P->unit_loop ? (R1Common&)au : (R1Common&)a1;
    a.x = x; a.h0 = h0; a.c0 = has_c ? c0 : nullptr; a.y = y; a.hT = hT; a.cT = has_c ? cT : nullptr;
    // What lies elsewhere while the kernel runs: host arrays; an input that an output overlaps (a CTA stores its last
    // states while another may still be reading the first ones; c0 given as cT is the exception, since a CTA reads
    // and writes its own units only); final states that overlap another output (copied after it, hT before cT).
    auto meets = [](const float* p, size_t n, const float* q, size_t m) { return p && q && n && m && p < q + m && q < p + n; };
    auto read_and_written = [&](const float* p, size_t n) { return meets(p, n, a.y, ny) || meets(p, n, a.hT, nh) || meets(p, n, a.cT, nc); };
    const bool move_x = host_io || read_and_written(a.x, nx), move_h0 = host_io || read_and_written(a.h0, nh);
    const bool move_c0 = host_io || (a.c0 != a.cT ? read_and_written(a.c0, nc) : meets(a.c0, nc, a.y, ny) || meets(a.c0, nc, a.hT, nh));
    const bool move_y = host_io, states_meet = meets(a.hT, nh, a.cT, nc);
    const bool move_hT = host_io || states_meet || meets(a.hT, nh, a.y, ny), move_cT = host_io || states_meet || meets(a.cT, nc, a.y, ny);
    {
        // (the states' copies have a place of their own from the start, so that a captured call can have them; a place
        // for x that was once used stays as long as the plan, for calls that were captured with it)
        float* d = P->d_states;
        float* dx = P->d_x;
        if (host_io) {
            const size_t need = nx + ny;
            if (need > P->stage_cap) {
                CSB_CUDA(cudaStreamSynchronize(st));
                cudaFree(P->d_stage); P->d_stage = nullptr; P->stage_cap = 0;
                CSB_CUDA(cudaMalloc((void**)&P->d_stage, need * 4));
                P->stage_cap = need;
            }
            dx = P->d_stage;
        } else if (move_x && nx > P->x_cap) {
            const size_t cap = std::max(nx, 2 * P->x_cap);
            CSB_CUDA(cudaMalloc((void**)&dx, cap * 4));
            P->own.p.push_back(dx);
            P->d_x = dx; P->x_cap = cap;
        }
        const cudaMemcpyKind kind = host_io ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
        auto in = [&](const float*& p, float* to, size_t n) -> cudaError_t {
            if (!p) return cudaSuccess;
            const cudaError_t e = cudaMemcpyAsync(to, p, n * 4, kind, st);
            p = to;
            return e;
        };
        if (move_x) CSB_CUDA(in(a.x, dx, nx));
        if (move_h0) CSB_CUDA(in(a.h0, d, nh));
        if (move_c0) CSB_CUDA(in(a.c0, d + nh, nc));
        if (move_y && a.y) a.y = dx + nx;
        if (move_hT && a.hT) a.hT = d + nh + nc;
        if (move_cT && a.cT) a.cT = d + 2 * nh + nc;
    }
    for (int l = 0; l < L; ++l) a.bias[l] = bias ? bias[l] : nullptr;
    a.T = (int)T; a.B = B;
    uint32_t extra = 0;
    barrier_test_hook(&extra, &a.limit_ns);
    a.never = extra ? 0x40000000u : 0u;
    *P->h_status = 0;
#ifdef CSB_PHASE_CLOCKS
    if (!g_r1_clocks) cudaMalloc((void**)&g_r1_clocks, 192 * 8 * 8);
    a.clocks = g_r1_clocks; g_r1_clock_ctas = P->n_ctas;
#endif
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)P->n_ctas); cfg.blockDim = dim3(kR1Threads); cfg.dynamicSmemBytes = P->smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    void* params[] = {P->unit_loop ? (void*)&au : (void*)&a1};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, P->kernel, params);
    if (e == cudaErrorCooperativeLaunchTooLarge) { set_error("cooperative launch too large"); return CSB_ERR_LAUNCH; }
    CSB_CUDA(e);
    const cudaMemcpyKind out_kind = host_io ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    if (move_y && y) CSB_CUDA(cudaMemcpyAsync(y, a.y, ny * 4, out_kind, st));
    if (move_hT && hT) CSB_CUDA(cudaMemcpyAsync(hT, a.hT, nh * 4, out_kind, st));
    if (move_cT && has_c && cT) CSB_CUDA(cudaMemcpyAsync(cT, a.cT, nc * 4, out_kind, st));
    if (host_io || !(flags & CSB_FLAG_ASYNC)) {
        CSB_CUDA(cudaStreamSynchronize(st));
        if (*P->h_status != 0) {
            set_error("the time-loop kernel gave up a bounded wait (code %u: %s)", *P->h_status,
                      *P->h_status == kDevBarrierTimeout ? "a vector from other CTAs" : "bulk copy");
            return CSB_ERR_TIMEOUT;
        }
    }
    return CSB_OK;
}

}  // namespace csb
