// LSTM and GRU layers at larger batch, one timestep at a time on tensor cores: what the time loop of csb_umma_rnn.cu does not
// take (more than 32 sequences, stacks that one grid does not hold, blocks whose width is not 16, 32 or a multiple of 64).
//
// With a batch of 16 or more the per-step product of Section 2.1, W . [u_t ; h_{t-1}] for all
// batch columns at once, is a dense contraction per block (kernel matrix times gathered inputs),
// which the batched product kernel runs on tensor cores.  The persistent time-loop kernel keeps
// that product on CUDA cores, so for these batches a step is issued as separate launches instead:
// the batched product (pack + tensor-core kernel) of every layer, then one small kernel with the
// gate arithmetic, which also routes h_t to where the next products read it.  The products of a
// layer read one buffer V_l = [u_t ; h_{t-1}] of shape [B, I_l + H]; the gate kernel of layer l
// writes h_t into the right part of V_l (for step t + 1) and into the left part of V_{l+1} (the
// layer above, same step) or into y, and the gate kernel of layer 0 also moves x_{t+1} in.
//
// Up to 32 product rows (LSTM: batch <= 32, GRU: batch <= 16) the fp32 buffers V_l do not exist at all:
// the gate arithmetic writes h_t, and that of layer 0 also x_{t+1}, straight into the packed binary16
// (hi, lo) input rows that the product kernel reads, transposed through shared memory so that the
// stores of a row are contiguous.  The layers then run as a wavefront: in tick k layer l does step k - l,
// which needs nothing newer than tick k - 1, so one product launch (the SMs shared between the layers) and
// one launch of gates serve all layers, and the fixed cost of the two is paid once per tick instead of once
// per layer and step.  Measured, two 2048-unit LSTM layers, 10x pruned, batch 32: 51 -> 29.6 us per step.
//
// GRU (reset gate applied after the recurrent product) needs the input part and the recurrent part
// of the candidate's pre-activation apart.  One product still does: V_l has 2B rows, row b holds
// [u_t ; 0] and row B + b holds [0 ; h_{t-1}], so row b of the product is W_x u and row B + b is W_h h.
// On the layouts of csb_umma.hpp the two parts are output rows of their own, and V_l has B rows.
#include <algorithm>
#include <list>
#include <memory>
#include <mutex>

#include "csb_host.hpp"
#include "csb_internal.hpp"
#include "csb_device.cuh"
#include "csb_gates.cuh"
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

struct StepPlan {
    std::vector<uint64_t> uids;
    int L = 0, B = 0, H = 0, gates = 0, device = -1;
    bool tiles = false, unpacked = false;   // what the environment asked for: the products on tcgen05, fp32 buffers for any batch
    int in_size[kMaxLayers] = {};
    float* d_v[kMaxLayers] = {};       // [B, in_size[l] + H] per layer (GRU: [2B, ...], input rows then recurrent rows)
    float* d_z = nullptr;              // [B, 4H] (GRU: [2B, 3H]) pre-activations; packed path: one such per layer
    SpmmStack stack;                   // packed path
    std::shared_ptr<UmmaStack> umma;   // the products run on these layouts (fp32 buffers only), one row per sequence for the GRU too
    float* d_c = nullptr;              // [L, B, H] cell state
    float* d_stage = nullptr;          // host-I/O staging of x and y
    size_t stage_cap = 0;
    // per layer the packed inputs of its product, one row of `pitch` bytes per column of W_l
    uint8_t* d_xp[kMaxLayers] = {};
    // packed path (at most 32 product rows): the fp32 h of every layer, and the layout of d_xp
    float* d_h = nullptr;              // [L, B, H]
    int pitch = 0, cap = 0;
    ~StepPlan() {
        for (float* p : d_v) cudaFree(p);
        for (uint8_t* p : d_xp) cudaFree(p);
        cudaFree(d_z); cudaFree(d_c); cudaFree(d_stage); cudaFree(d_h);
    }
};
static std::mutex g_step_mu;
static std::list<std::unique_ptr<StepPlan>> g_step_plans;

void drop_step_plans(const csb_matrix* A) {
    std::lock_guard<std::mutex> lk(g_step_mu);
    int prev = 0;
    cudaGetDevice(&prev);
    for (auto it = g_step_plans.begin(); it != g_step_plans.end();) {
        if (std::find((*it)->uids.begin(), (*it)->uids.end(), A->uid) != (*it)->uids.end()) {
            cudaSetDevice((*it)->device);
            it = g_step_plans.erase(it);
        } else ++it;
    }
    cudaSetDevice(prev);
}

// Gate arithmetic of one LSTM layer and step for the whole batch (Section 2.1):
//   c_t = s(z_f) c_{t-1} + s(z_i) tanh(z_g),  h_t = s(z_o) tanh(c_t),  rows of z stacked i, f, g, o.
// h_t goes to v_self[b, off_self + j] (this layer's next product), to v_next[b, j] (the layer
// above) when there is one, and to y_t[b, j] when asked.  With x_next the kernel also copies the
// next step's input rows into v0[b, 0 .. I).
__global__ void csb_lstm_gates_kernel(const float* __restrict__ Z, const float* __restrict__ bias, float* __restrict__ c,
                                      float* __restrict__ v_self, int ld_self, int off_self, float* __restrict__ v_next,
                                      int ld_next, float* __restrict__ y_t, const float* __restrict__ x_next, int I,
                                      float* __restrict__ v0, int ld0, int B, int H) {
    pdl_launch_dependents();
    pdl_wait();                                    // Z comes from the product in front
    const int n = B * H;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int b = e / H, j = e - b * H;
        const float* z = Z + (size_t)b * 4 * H;
        float zi = z[j], zf = z[H + j], zg = z[2 * H + j], zo = z[3 * H + j];
        if (bias) { zi += bias[j]; zf += bias[H + j]; zg += bias[2 * H + j]; zo += bias[3 * H + j]; }
        float cn = c[e];
        const float h = lstm_cell(zi, zf, zg, zo, cn);
        c[e] = cn;
        v_self[(size_t)b * ld_self + off_self + j] = h;
        if (v_next) v_next[(size_t)b * ld_next + j] = h;
        if (y_t) y_t[e] = h;
    }
    if (x_next) {
        const int nx = B * I;
        for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nx; e += gridDim.x * blockDim.x) {
            const int b = e / I, i = e - b * I;
            v0[(size_t)b * ld0 + i] = x_next[e];
        }
    }
}

// Gate arithmetic of one GRU layer and step (reset after the recurrent product):
//   r = s(zx_r + zh_r + b_r),  u = s(zx_z + zh_z + b_z),  n = tanh(zx_n + b_in + r (zh_n + b_hn)),
//   h_t = (1 - u) n + u h_{t-1};  zx = row b, zh = row B + b of Z [2B, 3H]; bias = b_r, b_z, b_in, b_hn.
// h_t goes to the recurrent rows of v_self (row B + b, columns off_self ..), to the input rows of
// v_next (row b) when there is a layer above, and to y_t; x_next as for the LSTM kernel.
// APART: the product itself has kept the candidate's parts apart, row b of Z [B, 4H] is r, z and the two parts, and v_self has
// one row per sequence.
template <bool APART>
__global__ void csb_gru_gates_kernel(const float* __restrict__ Z, const float* __restrict__ bias, float* __restrict__ v_self,
                                     int ld_self, int off_self, float* __restrict__ v_next, int ld_next, float* __restrict__ y_t,
                                     const float* __restrict__ x_next, int I, float* __restrict__ v0, int ld0, int B, int H) {
    pdl_launch_dependents();
    pdl_wait();                                    // Z comes from the product in front
    const int n = B * H;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int b = e / H, j = e - b * H;
        const float* zx = Z + (size_t)b * (APART ? 4 : 3) * H;
        const float* zh = Z + (size_t)(B + b) * 3 * H;
        float ar = zx[j], au = zx[H + j], nx = zx[2 * H + j], nh = APART ? zx[3 * H + j] : zh[2 * H + j];
        if (!APART) { ar += zh[j]; au += zh[H + j]; }
        if (bias) { ar += bias[j]; au += bias[H + j]; nx += bias[2 * H + j]; nh += bias[3 * H + j]; }
        float* hp = v_self + (size_t)(APART ? b : B + b) * ld_self + off_self + j;
        const float h = gru_cell(ar, au, nx, nh, *hp);
        *hp = h;
        if (v_next) v_next[(size_t)b * ld_next + j] = h;
        if (y_t) y_t[e] = h;
    }
    if (x_next) {
        const int nx = B * I;
        for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nx; e += gridDim.x * blockDim.x) {
            const int b = e / I, i = e - b * I;
            v0[(size_t)b * ld0 + i] = x_next[e];
        }
    }
}

// ---- the packed path (device functions in csb_gates.cuh) ----------------------------------------------
// Everything a sequence starts from, in one launch: the packed inputs of every layer, x_0 and h0 in
// them and the rest zero, and the running states.  A block takes 32 columns of a layer, the input
// columns first.  As separate clears, copies and packs it was half of the launches of a call of one
// step (two layers with states: 15, with the copies of the final states; 7 now, 41 us for 16 sequences
// on 2 x 900 units).
struct BeginArgs {
    const float* x; const float* h0; const float* c0;   // h0, c0: null = zeros; may be hs, c themselves
    float* hs; float* c;                                 // [L, B, H]; c null: no cell state
    uint8_t* xp[kMaxLayers];
    int in_size[kMaxLayers], end[kMaxLayers];            // end: first block behind the layer
    int pitch, cap, B, H, slot_h;                        // slot_h: first batch slot of the recurrent columns' inputs
};
__global__ void __launch_bounds__(256) csb_begin_kernel(const __grid_constant__ BeginArgs a) {
    __shared__ float tile[32][33];
    pdl_launch_dependents();
    int l = 0, first = 0;
    while ((int)blockIdx.x >= a.end[l]) first = a.end[l++];
    const int in_blocks = (a.in_size[l] + 31) / 32, blk = (int)blockIdx.x - first;
    const bool rec = blk >= in_blocks;
    const int n = rec ? a.H : a.in_size[l], c0 = (rec ? blk - in_blocks : blk) * 32;
    uint8_t* xp = a.xp[l] + (rec ? (size_t)a.in_size[l] * a.pitch : 0);
    uint4* rows = reinterpret_cast<uint4*>(xp + (size_t)c0 * a.pitch);
    for (int i = threadIdx.x; i < min(32, n - c0) * a.pitch / 16; i += blockDim.x) rows[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (rec) {
        const int tx = threadIdx.x & 31;
        const size_t at = (size_t)l * a.B * a.H + c0 + tx;
        for (int b = threadIdx.x >> 5; b < a.B; b += blockDim.x >> 5) {
            const size_t e = at + (size_t)b * a.H;
            const bool in = c0 + tx < n;
            const float h = in && a.h0 ? a.h0[e] : 0.f;
            tile[b][tx] = h;
            if (in) a.hs[e] = h;
            if (in && a.c) a.c[e] = a.c0 ? a.c0[e] : 0.f;
        }
        __syncthreads();
        if (a.h0) pack_tile(tile, min(32, n - c0), a.B, reinterpret_cast<uint8_t*>(rows), a.pitch, a.cap, a.slot_h, nullptr, 0);
    } else if (l == 0) {
        pack_columns(tile, a.x, (long long)n, a.B, n, c0, xp, a.pitch, a.cap, 0);
    }
}

// The gates of one tick: blocks [part, next part) take a layer's hidden units, 32 at a time and 8 batch
// columns each, the blocks behind the last part pack x_next [B, I] (the next input of layer 0) into
// rows of xp0.
struct GatePart {
    const float* Z; const float* bias; float* c; float* hs; uint8_t* xp_self; uint8_t* xp_next; float* y;
    int end;                                       // first block behind the part
};
struct GateArgs {
    GatePart part[kMaxLayers];
    const float* x_next; uint8_t* xp0;
    int n_parts, I, pitch, cap, B, H, b_tiles;
};
template <int GATES>
__global__ void __launch_bounds__(256) csb_gates_pack_kernel(const __grid_constant__ GateArgs a) {
    __shared__ float tile[32][33];
    pdl_launch_dependents();
    pdl_wait();                                    // Z comes from the product in front, which also still reads xp0
    int first = 0, p = 0;
    while (p < a.n_parts && (int)blockIdx.x >= a.part[p].end) first = a.part[p++].end;
    const int blk = (int)blockIdx.x - first;
    if (p < a.n_parts) {
        const GatePart& g = a.part[p];
        const int j0 = blk / a.b_tiles * 32, b0 = blk % a.b_tiles * 8, nb = min(8, a.B - b0);
        if (GATES == 4) lstm_gates_tile(tile, g.Z, g.bias, g.c, g.hs, g.xp_self, g.xp_next, g.y, a.pitch, a.cap, b0, nb, a.H, j0);
        else gru_gates_tile(tile, g.Z, g.bias, g.hs, g.xp_self, g.xp_next, g.y, a.pitch, a.cap, a.B, b0, nb, a.H, j0);
    } else {
        pack_columns(tile, a.x_next, (long long)a.I, a.B, a.I, blk * 32, a.xp0, a.pitch, a.cap, 0);
    }
}

static int env_flag(const char* name) {
    const char* v = getenv(name);
    return v && *v ? atoi(v) : 0;
}

bool rnn_stepwise_wanted(int gates, int L, const csb_matrix* const* W, int B) {
    if (env_flag("CSB_RNN_NO_STEPWISE")) return false;
    // from batch 16 always; from batch 8 when the layers are big enough for three launches per layer
    // and step to pay (measured: 591 k weights 24 -> 17 us per step, 25 k weights 9 -> 13)
    int64_t nnz = 0;
    for (int l = 0; l < L; ++l) nnz += W[l]->nnz;
    if (!(B >= 16 || (B >= 8 && nnz >= 100000))) return false;
    for (int l = 0; l < L; ++l)
        if (!spmm_mma_applicable(W[l], gates == 3 ? 2 * B : B)) return false;
    return true;
}

// Returns CSB_OK, an error, or 1 when the tensor-core plan of a layer does not fit (nothing the
// caller can see has been written then; the caller runs the persistent kernel instead).
int rnn_forward_stepwise(int gates, int L, const csb_matrix* const* W, const float* const* bias, const float* x, int64_t T, int B, int H,
                         const int* in_size, const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags,
                         void* stream) {
    StepPlan* P = nullptr;
    bool tiles = true;
    const bool unpacked = env_flag("CSB_RNN_STEP_UNPACKED") != 0;
    for (int l = 0; l < L; ++l) tiles = tiles && umma_applicable(W[l]);
    {
        std::lock_guard<std::mutex> lk(g_step_mu);
        for (auto& p : g_step_plans) {
            if (p->L != L || p->B != B || p->gates != gates || p->tiles != tiles || p->unpacked != unpacked) continue;
            bool same = true;
            for (int l = 0; l < L; ++l) same = same && p->uids[l] == W[l]->uid;
            if (same) { P = p.get(); break; }
        }
        if (!P) {
            std::unique_ptr<StepPlan> np(new StepPlan());
            np->L = L; np->B = B; np->H = H; np->gates = gates; np->device = W[0]->device; np->tiles = tiles; np->unpacked = unpacked;
            // The layouts of the time loop serve the fp32 buffers as well: its numbers bit for bit, and batches past 32 at the
            // speed of the bare product.
            const bool small = (gates == 3 ? 2 : 1) * B <= 32;
            if (!small || unpacked) {
                const int urc = umma_stack(gates, L, W, in_size, H, false, &np->umma);
                if (urc != CSB_OK) return urc;
            }
            const int rows_v = (gates == 3 && !np->umma ? 2 : 1) * B;
            const bool packed_path = small && !unpacked;
            const int pitch = spmm_pitch(spmm_nt(std::min(rows_v, 32)));
            if (packed_path) { np->pitch = pitch; np->cap = 8 * spmm_nt(rows_v); }
            for (int l = 0; l < L; ++l) {
                np->uids.push_back(W[l]->uid);
                np->in_size[l] = in_size[l];
                // (what is read of the packed inputs is written on the call's stream first, so they need no clearing here)
                CSB_CUDA(cudaMalloc((void**)&np->d_xp[l], np->umma ? umma_xp_bytes(np->umma->plan[l].windows) : (size_t)(in_size[l] + H) * pitch));
                if (!packed_path) CSB_CUDA(cudaMalloc((void**)&np->d_v[l], (size_t)rows_v * (in_size[l] + H) * 4));
            }
            const int rc = np->umma ? (int)CSB_OK : prepare_spmm_stack(L, W, std::min(rows_v, 32), &np->stack);
            if (rc != CSB_OK) return rc;
            if (packed_path) CSB_CUDA(cudaMalloc((void**)&np->d_h, (size_t)L * B * H * 4));
            CSB_CUDA(cudaMalloc((void**)&np->d_z, (size_t)(packed_path ? L : 1) * rows_v * (np->umma ? 4 : gates) * H * 4));
            if (gates == 4) CSB_CUDA(cudaMalloc((void**)&np->d_c, (size_t)L * B * H * 4));
            P = np.get();
            g_step_plans.push_back(std::move(np));
        }
    }
    note_recurrent_path(P->pitch ? kPathStepsPacked : kPathSteps);
    cudaStream_t st = (cudaStream_t)stream;
    const bool host_io = (flags & CSB_FLAG_HOST_IO) != 0;
    const int I0 = in_size[0];
    const size_t nx = (size_t)T * B * I0, ny = (size_t)T * B * H, ns = (size_t)L * B * H;
    const float* dx = x;
    float* dy = y;
    if (host_io) {
        const size_t need = nx + (y ? ny : 0);
        if (need > P->stage_cap) {
            CSB_CUDA(cudaStreamSynchronize(st));
            cudaFree(P->d_stage); P->d_stage = nullptr; P->stage_cap = 0;
            CSB_CUDA(cudaMalloc((void**)&P->d_stage, need * 4));
            P->stage_cap = need;
        }
        CSB_CUDA(cudaMemcpyAsync(P->d_stage, x, nx * 4, cudaMemcpyHostToDevice, st));
        dx = P->d_stage;
        dy = y ? P->d_stage + nx : nullptr;
    }
    const cudaMemcpyKind in_kind = host_io ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    const cudaMemcpyKind out_kind = host_io ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    const size_t hrow = (size_t)H * 4;
    const bool gru = gates == 3;
    const bool apart_rows = gru && !P->umma;            // input and recurrent rows of their own
    const int vrows = apart_rows ? 2 * B : B;           // rows of V_l and of the product
    if (P->pitch) {
        // ---- packed path: the gate kernels feed the products' packed inputs directly
        const int pitch = P->pitch, cap = P->cap;
        // The states run in the caller's final-state arrays where nothing else lies there, else in the plan's
        auto apart = [](const float* p, size_t n, const float* q, size_t m) { return !p || !q || p + n <= q || q + m <= p; };
        const size_t nx1 = (size_t)T * B * I0;
        const bool direct = !host_io && apart(hT, ns, cT, ns);
        const bool own_h = !(direct && hT && apart(hT, ns, x, nx1) && apart(hT, ns, y, ny) && apart(hT, ns, c0, ns) && (h0 == hT || apart(hT, ns, h0, ns)));
        const bool own_c = !(direct && cT && apart(cT, ns, x, nx1) && apart(cT, ns, y, ny) && apart(cT, ns, h0, ns) && (c0 == cT || apart(cT, ns, c0, ns)));
        float* hs = own_h ? P->d_h : hT;
        float* cs = gru ? nullptr : own_c ? P->d_c : cT;
        BeginArgs ba{};
        ba.x = dx; ba.h0 = h0; ba.c0 = c0; ba.hs = hs; ba.c = cs;
        if (host_io) {
            if (h0) { CSB_CUDA(cudaMemcpyAsync(hs, h0, ns * 4, in_kind, st)); ba.h0 = hs; }
            if (c0 && cs) { CSB_CUDA(cudaMemcpyAsync(cs, c0, ns * 4, in_kind, st)); ba.c0 = cs; }
        }
        ba.pitch = pitch; ba.cap = cap; ba.B = B; ba.H = H; ba.slot_h = gru ? B : 0;
        int begin_blocks = 0;
        for (int l = 0; l < L; ++l) {
            ba.xp[l] = P->d_xp[l]; ba.in_size[l] = in_size[l];
            begin_blocks += (in_size[l] + 31) / 32 + (H + 31) / 32;
            ba.end[l] = begin_blocks;
        }
        csb_begin_kernel<<<begin_blocks, 256, 0, st>>>(ba);
        CSB_CUDA(cudaGetLastError());
        const int h_tiles = (H + 31) / 32, b_tiles = (B + 7) / 8, x_blocks = (I0 + 31) / 32;
        float* Z[kMaxLayers];
        for (int l = 0; l < L; ++l) Z[l] = P->d_z + (size_t)l * vrows * gates * H;
        for (int64_t k = 0; k < T + L - 1; ++k) {
            // the layers with a step in this tick are neighbours
            const int l0 = (int)std::max<int64_t>(0, k - T + 1), l1 = (int)std::min<int64_t>(L, k + 1);
            const int rc = launch_spmm_stack(P->stack, l0, l1, W, P->d_xp, Z, vrows, (int64_t)gates * H, stream);
            if (rc != CSB_OK) return rc;
            GateArgs a{};
            a.n_parts = l1 - l0; a.I = I0; a.pitch = pitch; a.cap = cap; a.B = B; a.H = H; a.b_tiles = b_tiles;
            int blocks = 0;
            for (int l = l0; l < l1; ++l) {
                GatePart& g = a.part[l - l0];
                const int64_t t = k - l;
                g.Z = Z[l]; g.bias = bias ? bias[l] : nullptr; g.c = gru ? nullptr : cs + (size_t)l * B * H; g.hs = hs + (size_t)l * B * H;
                g.xp_self = P->d_xp[l] + (size_t)in_size[l] * pitch; g.xp_next = l + 1 < L ? P->d_xp[l + 1] : nullptr;
                g.y = (l == L - 1 && dy) ? dy + (size_t)t * B * H : nullptr;
                blocks += h_tiles * b_tiles;
                g.end = blocks;
            }
            if (k + 1 < T) { a.x_next = dx + (size_t)(k + 1) * B * I0; a.xp0 = P->d_xp[0]; blocks += x_blocks; }
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = 0;
            cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 1;
            CSB_CUDA(cudaLaunchKernelEx(&cfg, gru ? csb_gates_pack_kernel<3> : csb_gates_pack_kernel<4>, a));
            CSB_CUDA(cudaGetLastError());
        }
        if (hT && own_h) CSB_CUDA(cudaMemcpyAsync(hT, hs, ns * 4, out_kind, st));
        if (cT && !gru && own_c) CSB_CUDA(cudaMemcpyAsync(cT, cs, ns * 4, out_kind, st));
        if (host_io && y) CSB_CUDA(cudaMemcpyAsync(y, dy, ny * 4, cudaMemcpyDeviceToHost, st));
        if (host_io || !(flags & CSB_FLAG_ASYNC)) {
            CSB_CUDA(cudaStreamSynchronize(st));
            for (int l = 0; l < L; ++l)
                if (W[l]->product.h_status && *W[l]->product.h_status != 0) {
                    set_error("a product kernel of layer %d gave up a bounded wait (code %u)", l, *W[l]->product.h_status);
                    return CSB_ERR_TIMEOUT;
                }
        }
        return CSB_OK;
    }
    // V_l = [u_0 ; h_{-1}]: h0 (or zeros) on the right, x_0 on the left of layer 0.  GRU: the
    // recurrent rows (B ..) carry h and zeros on the left, the input rows zeros on the right.
    for (int l = 0; l < L; ++l) {
        const int ld = in_size[l] + H;
        float* hpart = P->d_v[l] + (apart_rows ? (size_t)B * ld : 0) + in_size[l];
        if (apart_rows) CSB_CUDA(cudaMemsetAsync(P->d_v[l], 0, (size_t)vrows * ld * 4, st));
        if (h0) CSB_CUDA(cudaMemcpy2DAsync(hpart, (size_t)ld * 4, h0 + (size_t)l * B * H, hrow, hrow, B, in_kind, st));
        else if (!apart_rows) CSB_CUDA(cudaMemset2DAsync(hpart, (size_t)ld * 4, 0, hrow, B, st));
    }
    CSB_CUDA(cudaMemcpy2DAsync(P->d_v[0], (size_t)(I0 + H) * 4, dx, (size_t)I0 * 4, (size_t)I0 * 4, B, cudaMemcpyDeviceToDevice, st));
    if (!gru) {
        if (c0) CSB_CUDA(cudaMemcpyAsync(P->d_c, c0, ns * 4, in_kind, st));
        else CSB_CUDA(cudaMemsetAsync(P->d_c, 0, ns * 4, st));
    }

    const int threads = 256;
    const int blocks = std::max(1, std::min(1024, (B * std::max(H, I0) + threads - 1) / threads));
    for (int64_t t = 0; t < T; ++t) {
        for (int l = 0; l < L; ++l) {
            const int ld = in_size[l] + H;
            int rc = product_gave_up(W[l]);
            if (rc != CSB_OK) return rc;
            rc = P->umma ? launch_umma_fp32(W[l], &P->umma->plan[l], P->d_xp[l], P->d_v[l], ld, vrows, P->d_z, (int64_t)4 * H, st)
                         : launch_spmm_stack_fp32(P->stack, l, W[l], P->d_xp[l], P->d_v[l], ld, vrows, P->d_z, (int64_t)gates * H, stream);
            if (rc != CSB_OK) return rc;
            const bool top = l == L - 1;
            const float* x_next = (l == 0 && t + 1 < T) ? dx + (size_t)(t + 1) * B * I0 : nullptr;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = 0;
            cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 1;
            const float* bl = bias ? bias[l] : nullptr;
            float* vn = top ? nullptr : P->d_v[l + 1];
            const int ldn = top ? 0 : in_size[l + 1] + H;
            float* yt = (top && dy) ? dy + (size_t)t * B * H : nullptr;
            if (gru)
                CSB_CUDA(cudaLaunchKernelEx(&cfg, P->umma ? csb_gru_gates_kernel<true> : csb_gru_gates_kernel<false>, (const float*)P->d_z, bl, P->d_v[l], ld, in_size[l], vn, ldn, yt,
                                            x_next, I0, P->d_v[0], I0 + H, B, H));
            else
                CSB_CUDA(cudaLaunchKernelEx(&cfg, csb_lstm_gates_kernel, (const float*)P->d_z, bl, P->d_c + (size_t)l * B * H, P->d_v[l], ld,
                                            in_size[l], vn, ldn, yt, x_next, I0, P->d_v[0], I0 + H, B, H));
            CSB_CUDA(cudaGetLastError());
        }
    }
    if (hT)
        for (int l = 0; l < L; ++l)
            CSB_CUDA(cudaMemcpy2DAsync(hT + (size_t)l * B * H, hrow, P->d_v[l] + (apart_rows ? (size_t)B * (in_size[l] + H) : 0) + in_size[l],
                                       (size_t)(in_size[l] + H) * 4, hrow, B, out_kind, st));
    if (cT && !gru) CSB_CUDA(cudaMemcpyAsync(cT, P->d_c, ns * 4, out_kind, st));
    if (host_io && y) CSB_CUDA(cudaMemcpyAsync(y, dy, ny * 4, cudaMemcpyDeviceToHost, st));
    if (host_io || !(flags & CSB_FLAG_ASYNC)) {
        CSB_CUDA(cudaStreamSynchronize(st));
        for (int l = 0; l < L; ++l)
            if (W[l]->product.h_status && *W[l]->product.h_status != 0) {
                set_error("a product kernel of layer %d gave up a bounded wait (code %u)", l, *W[l]->product.h_status);
                return CSB_ERR_TIMEOUT;
            }
    }
    return CSB_OK;
}

}  // namespace csb
