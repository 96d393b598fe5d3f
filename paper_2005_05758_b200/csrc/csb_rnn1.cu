// Batch-1 time loop of the recurrent cells (LSTM, GRU, LSTMP, Li-GRU, reset-before GRU): one
// cooperative launch per sequence (Section 2.1 of the paper: per step a CSB product with
// [u_t ; h_{t-1}], then the element-wise gate arithmetic, the c / h "context link" feeding the next step).
//
// A CTA owns a range of hidden units of one layer (csb_rnn1.hpp); its weights stay in shared memory.
// What bounds a step is latency: the exchange of h_t between CTAs, then the chain gather -> product ->
// sum -> gates.  So
//   * a vector crosses CTAs as 16-byte words of three values and the number of their step, written
//     and read with single 16-byte accesses (relaxed, 128-bit atomic): a reader that sees the step
//     it waits for also holds the values.  No fence, no counter, no grid barrier; layers run as a
//     dataflow pipeline.  Step numbers go on from call to call (a word per CTA keeps the count), so
//     nothing is cleared between calls.  A vector stays for 32 steps; every 8 steps a layer checks
//     that the layer above has read what it is about to overwrite;
//   * the product over the input part [u_t] is done while h_{t-1} is on its way;
//   * the product is a plain loop: per pair of slots a lane reads 16 bytes of weights, two places and
//     two times four gathered inputs, and adds into one register pair; every thread works for one
//     row, so there is no scatter, and a row's threads meet once, in the gate arithmetic;
//   * a unit's gates sit on four neighbouring lanes, so the gate arithmetic needs no further barrier.
// LSTMP and the reset-before GRU have a second product in the step (the projection; the candidate's):
// what it reads (o * tanh(c); r * h) crosses the CTAs of the layer in the same way.
//
// Initial states, bias, x, y and final states are read and written in place, so a call is one launch.
#include <cstdlib>
#include <list>
#include <memory>
#include <mutex>

#include "csb_rnn1.hpp"
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

struct R1Args {
    const uint8_t* images;
    const R1Cta* ctas;
    const float* x; const float* h0; const float* c0;
    float* y; float* hT; float* cT;
    const float* bias[kMaxLayers];
    int in_size[kMaxLayers];
    const uint32_t* wmap[2][kMaxLayers];       // unit0 | units << 16 of every exchange word
    int words[2][kMaxLayers];
    uint4* ex[2][kMaxLayers];                  // [kR1Ring][words]
    uint32_t* epoch;                           // per CTA: step numbers used so far
    uint32_t* progress;                        // per layer: blocks of kR1Block input steps read, summed over its CTAs, never cleared
    int layer_ctas[kMaxLayers];
    uint32_t* status;
    unsigned long long limit_ns;
    uint32_t never;                            // test hook: wait for step numbers that never come
    int T, H, S, L;
    uint32_t xg[2][2], vu, vr, vm, part, misc; // shared-memory offsets behind the image
};

__device__ __forceinline__ uint4 ld_word(const uint4* p) {
    uint64_t a, b;
    asm volatile("{\n\t.reg .b128 r;\n\tld.relaxed.gpu.global.b128 r, [%2];\n\tmov.b128 {%0, %1}, r;\n\t}" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ void st_word(uint4* p, uint4 v) {
    const uint64_t a = (uint64_t)v.x | ((uint64_t)v.y << 32), b = (uint64_t)v.z | ((uint64_t)v.w << 32);
    asm volatile("{\n\t.reg .b128 r;\n\tmov.b128 r, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], r;\n\t}" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)), "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 half2_to_float2(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }
__device__ __forceinline__ float logistic(float a) { return 1.f / (1.f + expf(-a)); }

// This thread's slots of one part of a product: `pairs` rounds of two slots, [round][lane].
template <typename T>
__device__ __forceinline__ float walk(const uint4* w, const uint32_t* places, int pairs, const uint8_t* xg) {
    float2 a = make_float2(0.f, 0.f), b = make_float2(0.f, 0.f);
    constexpr int kStride = sizeof(T) == 2 ? 32 : 64;
#pragma unroll 4
    for (int i = 0; i < pairs; ++i) {
        const uint32_t o = places[i * 32];
        const float4 x0 = *reinterpret_cast<const float4*>(xg + (o & 0xffffu)), x1 = *reinterpret_cast<const float4*>(xg + (o >> 16));
        if (sizeof(T) == 2) {
            const uint4 v = w[i * kStride];
            a = fma2(half2_to_float2(v.x), make_float2(x0.x, x0.y), a);
            b = fma2(half2_to_float2(v.y), make_float2(x0.z, x0.w), b);
            a = fma2(half2_to_float2(v.z), make_float2(x1.x, x1.y), a);
            b = fma2(half2_to_float2(v.w), make_float2(x1.z, x1.w), b);
        } else {
            const float4 v0 = *reinterpret_cast<const float4*>(w + i * kStride), v1 = *reinterpret_cast<const float4*>(w + i * kStride + 32);
            a = fma2(make_float2(v0.x, v0.y), make_float2(x0.x, x0.y), a);
            b = fma2(make_float2(v0.z, v0.w), make_float2(x0.z, x0.w), b);
            a = fma2(make_float2(v1.x, v1.y), make_float2(x1.x, x1.y), a);
            b = fma2(make_float2(v1.z, v1.w), make_float2(x1.z, x1.w), b);
        }
    }
    return (a.x + a.y) + (b.x + b.y);
}

// The pairs of the recurrent part that stay in registers for the whole sequence.
template <typename T, int N> struct RegPairs {
    static constexpr int kN = N, kV = sizeof(T) == 2 ? 1 : 2;
    uint4 w[kN][kV];
    uint32_t o[kN];
    __device__ __forceinline__ void load(const uint8_t* img, const R1Op& d, int warp, int lane) {
#pragma unroll
        for (int i = 0; i < kN; ++i) {
#pragma unroll
            for (int v = 0; v < kV; ++v) w[i][v] = __ldg(reinterpret_cast<const uint4*>(img + d.reg_off) + ((warp * kN + i) * kV + v) * 32 + lane);
            o[i] = __ldg(reinterpret_cast<const uint32_t*>(img + d.reg_places) + (warp * kN + i) * 32 + lane);
        }
    }
    __device__ __forceinline__ float walk(const uint8_t* xg) const {
        float2 a = make_float2(0.f, 0.f), b = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < kN; ++i) {
            const float4 x0 = *reinterpret_cast<const float4*>(xg + (o[i] & 0xffffu)), x1 = *reinterpret_cast<const float4*>(xg + (o[i] >> 16));
            const uint4 v = w[i][0], u = w[i][kV - 1];
            if (sizeof(T) == 2) {
                a = fma2(half2_to_float2(v.x), make_float2(x0.x, x0.y), a);
                b = fma2(half2_to_float2(v.y), make_float2(x0.z, x0.w), b);
                a = fma2(half2_to_float2(v.z), make_float2(x1.x, x1.y), a);
                b = fma2(half2_to_float2(v.w), make_float2(x1.z, x1.w), b);
            } else {
                a = fma2(make_float2(__uint_as_float(v.x), __uint_as_float(v.y)), make_float2(x0.x, x0.y), a);
                b = fma2(make_float2(__uint_as_float(v.z), __uint_as_float(v.w)), make_float2(x0.z, x0.w), b);
                a = fma2(make_float2(__uint_as_float(u.x), __uint_as_float(u.y)), make_float2(x1.x, x1.y), a);
                b = fma2(make_float2(__uint_as_float(u.z), __uint_as_float(u.w)), make_float2(x1.z, x1.w), b);
            }
        }
        return (a.x + a.y) + (b.x + b.y);
    }
};

// The kept inputs of a part's blocks, four a thread: xg[i] = v[idx[i]] (padding indices point at a zero).
__device__ __forceinline__ void gather(const uint16_t* idx, int quads, const float* v, float* xg) {
    for (int q = threadIdx.x; q < quads; q += kR1Threads) {
        const uint2 i = reinterpret_cast<const uint2*>(idx)[q];
        float4 r;
        r.x = v[i.x & 0xffffu]; r.y = v[i.x >> 16];
        r.z = v[i.y & 0xffffu]; r.w = v[i.y >> 16];
        reinterpret_cast<float4*>(xg)[q] = r;
    }
}

template <typename T, int CELL>
__global__ void __launch_bounds__(kR1Threads, 1) csb_rnn1_kernel(const __grid_constant__ R1Args a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int OPS = CELL == kR1Lstmp || CELL == kR1GruRb ? 2 : 1;
    constexpr int G0 = CELL == kR1Lstm || CELL == kR1Lstmp ? 4 : CELL == kR1Gru ? 3 : 2;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const R1Cta me = a.ctas[blockIdx.x];
    const int layer = me.layer, I = a.in_size[layer], S = a.S, H = a.H, T_ = a.T;
    float* vu = reinterpret_cast<float*>(smem + a.vu);
    float* vr = reinterpret_cast<float*>(smem + a.vr);
    float* vm = reinterpret_cast<float*>(smem + a.vm);
    float2* part = reinterpret_cast<float2*>(smem + a.part);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + a.misc);
    volatile int* s_ok = reinterpret_cast<volatile int*>(smem + a.misc + 8);
    const uint8_t* img = smem;

    // ---- weights, initial state, first input
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
        mbar_expect_tx(bar, me.smem_bytes);
        const uint8_t* src = a.images + (size_t)me.off16 * 16;
        for (uint32_t off = 0; off < me.smem_bytes; off += 16384u) bulk_g2s(smem + off, src + off, min(16384u, me.smem_bytes - off), bar);
        *s_ok = 1;
    }
    for (int i = tid; i <= S; i += kR1Threads) vr[i] = i < S && a.h0 ? __ldg(a.h0 + (size_t)layer * S + i) : 0.f;
    for (int i = tid; i <= I; i += kR1Threads) vu[i] = i < I && layer == 0 ? __ldg(a.x + i) : 0.f;
    if (OPS == 2 && tid == 0) vm[H] = 0.f;
    const uint32_t base = a.epoch[blockIdx.x] + 1u;        // the step number of step 0
    uint32_t above0 = 0;                                   // the progress of the layer above when this call began
    if (layer + 1 < a.L) above0 = ld_relaxed(a.progress + layer + 1);
    __syncthreads();
    bool ok = mbar_wait_bounded(bar, 0);
    if (!ok) *(volatile uint32_t*)a.status = (uint32_t)kDevCopyTimeout;
    if (!__syncthreads_and(ok)) {
        if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
        return;
    }

    // ---- what stays the same over the steps
    const R1Header* hd = reinterpret_cast<const R1Header*>(img);
    constexpr int kRegPairs = (sizeof(T) == 2 ? 4 : 2) / OPS;     // r1_reg_pairs()
    RegPairs<T, kRegPairs> regs[OPS];
    struct Walk { const uint4* w[2]; const uint32_t* o[2]; int n[2]; } wk[OPS];
    struct Gate { int u, t0, k; bool on; float bias; } gt[OPS];
    const int j = lane >> 2, g = lane & 3;
#pragma unroll
    for (int op = 0; op < OPS; ++op) {
        const R1Op& d = hd->op[op];
        regs[op].load(a.images + (size_t)me.off16 * 16, d, warp, lane);
        const uint4 wd = reinterpret_cast<const uint4*>(img + d.warp_off)[warp];
        wk[op].w[0] = reinterpret_cast<const uint4*>(img) + wd.x + lane;
        wk[op].w[1] = wk[op].w[0] + (size_t)wd.z * (sizeof(T) == 2 ? 32 : 64);
        wk[op].o[0] = reinterpret_cast<const uint32_t*>(img + wd.y) + lane;
        wk[op].o[1] = wk[op].o[0] + (size_t)wd.z * 32;
        wk[op].n[0] = (int)wd.z; wk[op].n[1] = (int)wd.w;
        // gate lanes: four per unit, six units per warp
        const int gates = op == 0 ? G0 : 1, u = warp * kR1WarpUnits + j;
        gt[op].u = (int)d.unit0 + u;
        gt[op].on = j < kR1WarpUnits && u < (int)d.units;
        // GRU: lanes 2 and 3 take the input and the hidden part of the candidate's row
        const int row_g = CELL == kR1Gru ? min(g, 2) : g;
        const bool has = gt[op].on && row_g < gates;
        const uint32_t row = has ? reinterpret_cast<const uint32_t*>(img + d.rows_off)[row_g * (int)d.units + u] : 0u;
        gt[op].t0 = (int)(row & 0xffffu); gt[op].k = (int)(row >> 16);
        const float* bl = a.bias[layer];
        gt[op].bias = 0.f;
        if (bl && gt[op].on) {
            if (op == 0 && g < (CELL == kR1Gru ? 4 : G0)) gt[op].bias = __ldg(bl + (size_t)g * H + gt[op].u);
            if (op == 1 && CELL == kR1GruRb && g == 0) gt[op].bias = __ldg(bl + (size_t)2 * H + gt[op].u);
        }
    }
    float c_state = 0.f;                                   // LSTM, LSTMP: cell state of the lanes' unit
    if ((CELL == kR1Lstm || CELL == kR1Lstmp) && gt[0].on && a.c0) c_state = __ldg(a.c0 + (size_t)layer * H + gt[0].u);

    // ---- the exchange.  Words are asked for early (poll_issue) and looked at late (poll_take).
    auto slot = [&](int e, int l, int t) { return a.ex[e][l] + (size_t)(t & (kR1Ring - 1)) * a.words[e][l]; };
    auto poll_issue = [&](uint4 (&w)[kR1Words], const uint4* src, int n) {
#pragma unroll
        for (int q = 0; q < kR1Words; ++q)
            if (tid + q * kR1Threads < n) w[q] = ld_word(src + tid + q * kR1Threads);
    };
    auto poll_take = [&](uint4 (&w)[kR1Words], const uint4* src, int n, const uint32_t* map, uint32_t want, float* dst) {
        want += a.never;
#pragma unroll
        for (int q = 0; q < kR1Words; ++q) {
            const int i = tid + q * kR1Threads;
            if (i >= n) continue;
            unsigned long long t0 = 0;
            unsigned int spins = 0;
            while (w[q].w != want) {
                if (*s_ok == 0) { ok = false; break; }     // another thread has given up
                if ((++spins & 63u) == 0) {
                    const unsigned long long now = global_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > a.limit_ns) { *(volatile uint32_t*)a.status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; ok = false; break; }
                }
                w[q] = ld_word(src + i);
            }
            const uint32_t m = __ldg(map + i);
            float* p = dst + (m & 0xffffu);
            p[0] = __uint_as_float(w[q].x);
            if ((m >> 16) > 1) p[1] = __uint_as_float(w[q].y);
            if ((m >> 16) > 2) p[2] = __uint_as_float(w[q].z);
        }
    };
    // The gate lanes' units to the other CTAs: two words of three units per warp.
    auto publish = [&](int e, int op, float v, int t) {
        const float v1 = __shfl_down_sync(0xffffffffu, v, 4), v2 = __shfl_down_sync(0xffffffffu, v, 8);
        if (gt[op].on && g == 0 && (j == 0 || j == 3))
            st_word(slot(e, layer, t) + hd->op[op].word0 + warp * 2 + j / 3,
                    make_uint4(__float_as_uint(v), __float_as_uint(v1), __float_as_uint(v2), base + (uint32_t)t));
    };
    // The sum of a gate lane's row over its threads.
    auto row_sum = [&](int op) {
        float s = 0.f;
        for (int i = 0; i < gt[op].k; ++i) {
            const float2 p = part[gt[op].t0 + i];
            s += CELL == kR1Gru ? (g == 3 ? p.y : g == 2 ? p.x : p.x + p.y) : p.x;
        }
        return s;
    };
    const bool gate_warp0 = warp * kR1WarpUnits < (int)hd->op[0].units, gate_warp1 = OPS == 2 && warp * kR1WarpUnits < (int)hd->op[OPS - 1].units;
    const int below = layer - 1;
    uint4 wr[kR1Words] = {}, wi[kR1Words] = {};
    if (layer > 0) {
        poll_issue(wi, slot(0, below, 0), a.words[0][below]);
        poll_take(wi, slot(0, below, 0), a.words[0][below], a.wmap[0][below], base, vu);
    }
    __syncthreads();

    for (int t = 0; t < T_; ++t) {
        const bool more = t + 1 < T_;
        // u_t lies in vu.  Ask for the state of the step before; the input part of the product meanwhile.
        const uint4* rec_src = slot(0, layer, t - 1);
        if (t > 0) poll_issue(wr, rec_src, a.words[0][layer]);
        gather(reinterpret_cast<const uint16_t*>(img + hd->op[0].gather_off[0]), hd->op[0].quads[0], vu, reinterpret_cast<float*>(smem + a.xg[0][0]));
        if (CELL == kR1GruRb)
            gather(reinterpret_cast<const uint16_t*>(img + hd->op[OPS - 1].gather_off[0]), hd->op[OPS - 1].quads[0], vu, reinterpret_cast<float*>(smem + a.xg[1][0]));
        float x_next[4];
        if (layer == 0 && more) {
#pragma unroll
            for (int q = 0; q < 4; ++q) if (tid + q * kR1Threads < I) x_next[q] = __ldg(a.x + (size_t)(t + 1) * I + tid + q * kR1Threads);
        }
        __syncthreads();
        if (layer > 0 && tid == 0 && (t & (kR1Block - 1)) == kR1Block - 1) atomicAdd(a.progress + layer, 1u);   // u up to step t has been read
        const float in0 = walk<T>(wk[0].w[0], wk[0].o[0], wk[0].n[0], smem + a.xg[0][0]);
        float in1 = 0.f;
        if (CELL == kR1GruRb) in1 = walk<T>(wk[OPS - 1].w[0], wk[OPS - 1].o[0], wk[OPS - 1].n[0], smem + a.xg[1][0]);
        if (t > 0) poll_take(wr, rec_src, a.words[0][layer], a.wmap[0][layer], base + (uint32_t)(t - 1), vr);
        if (more) {
            // every thread is past reading vu: the next input frame moves in; the layer below is asked for its next state
            if (layer == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) if (tid + q * kR1Threads < I) vu[tid + q * kR1Threads] = x_next[q];
                for (int i = tid + 4 * kR1Threads; i < I; i += kR1Threads) vu[i] = __ldg(a.x + (size_t)(t + 1) * I + i);
            } else poll_issue(wi, slot(0, below, t + 1), a.words[0][below]);
        }
        if (!__syncthreads_and(ok)) break;
        gather(reinterpret_cast<const uint16_t*>(img + hd->op[0].gather_off[1]), hd->op[0].quads[1], vr, reinterpret_cast<float*>(smem + a.xg[0][1]));
        __syncthreads();
        const float rec0 = regs[0].walk(smem + a.xg[0][1]) + walk<T>(wk[0].w[1], wk[0].o[1], wk[0].n[1], smem + a.xg[0][1]);
        part[tid] = CELL == kR1Gru ? make_float2(in0, rec0) : make_float2(in0 + rec0, 0.f);
        // before the slots of steps t .. t + 7 are overwritten, the layer above must have read what they
        // hold, steps up to t - 25.  Only the sum over its CTAs of the blocks of 8 they have read is kept:
        // CTAs of one layer are never more than two steps apart, so while one has not finished block k
        // none of the others has finished block k + 1, and the sum is below n k.
        if (layer + 1 < a.L && t >= kR1Ring && (t & (kR1Block - 1)) == 0 && tid == 0) {
            const uint32_t need = (uint32_t)a.layer_ctas[layer + 1] * (uint32_t)((t - kR1Ring + kR1Block) / kR1Block);
            unsigned long long t0 = 0;
            unsigned int spins = 0;
            while (ld_relaxed(a.progress + layer + 1) - above0 < need) {
                if ((++spins & 63u) == 0) {
                    const unsigned long long now = global_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > a.limit_ns) { *(volatile uint32_t*)a.status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; ok = false; break; }
                }
            }
        }
        if (!__syncthreads_and(ok)) break;
        // ---- gates
        float zg = 0.f;                                    // reset-before GRU: the update gate, on the unit's lane 1
        if (gate_warp0) {
            float z = row_sum(0) + gt[0].bias;
            const int l0 = lane & ~3;
            float h = 0.f;
            if (CELL == kR1Lstm || CELL == kR1Lstmp) {
                z = g == 2 ? tanhf(z) : logistic(z);
                const float zi = __shfl_sync(0xffffffffu, z, l0), zf = __shfl_sync(0xffffffffu, z, l0 + 1);
                const float zc = __shfl_sync(0xffffffffu, z, l0 + 2), zo = __shfl_sync(0xffffffffu, z, l0 + 3);
                c_state = zf * c_state + zi * zc;
                h = zo * tanhf(c_state);
                if (!more && a.cT && gt[0].on && g == 0) a.cT[(size_t)layer * H + gt[0].u] = c_state;
            } else if (CELL == kR1Gru) {
                if (g < 2) z = logistic(z);
                const float r = __shfl_sync(0xffffffffu, z, l0), zz = __shfl_sync(0xffffffffu, z, l0 + 1);
                const float ni = __shfl_sync(0xffffffffu, z, l0 + 2), nh = __shfl_sync(0xffffffffu, z, l0 + 3);
                const float n = tanhf(ni + r * nh), hp = gt[0].on ? vr[gt[0].u] : 0.f;
                h = (1.f - zz) * n + zz * hp;
            } else if (CELL == kR1Ligru) {
                if (g == 0) z = logistic(z);
                const float zz = __shfl_sync(0xffffffffu, z, l0), cand = fmaxf(__shfl_sync(0xffffffffu, z, l0 + 1), 0.f);
                const float hp = gt[0].on ? vr[gt[0].u] : 0.f;
                h = zz * hp + (1.f - zz) * cand;
            } else {
                z = logistic(z);
                zg = __shfl_sync(0xffffffffu, z, l0 + 1);
                h = __shfl_sync(0xffffffffu, z, l0) * (gt[0].on ? vr[gt[0].u] : 0.f);     // r * h_{t-1}
            }
            if (OPS == 2) publish(1, 0, h, t);
            else {
                if (more || layer + 1 < a.L) publish(0, 0, h, t);
                if (gt[0].on && g == 0) {
                    if (layer == a.L - 1 && a.y) a.y[(size_t)t * S + gt[0].u] = h;
                    if (!more && a.hT) a.hT[(size_t)layer * S + gt[0].u] = h;
                }
            }
        }
        if (OPS == 2) {
            // ---- second product of the step: what the first one gave, from every CTA of the layer
            const uint4* src = slot(1, layer, t);
            poll_issue(wr, src, a.words[1][layer]);
            poll_take(wr, src, a.words[1][layer], a.wmap[1][layer], base + (uint32_t)t, vm);
            if (!__syncthreads_and(ok)) break;
            gather(reinterpret_cast<const uint16_t*>(img + hd->op[1].gather_off[1]), hd->op[1].quads[1], vm, reinterpret_cast<float*>(smem + a.xg[1][1]));
            __syncthreads();
            part[tid] = make_float2(in1 + (regs[OPS - 1].walk(smem + a.xg[1][1]) + walk<T>(wk[OPS - 1].w[1], wk[OPS - 1].o[1], wk[OPS - 1].n[1], smem + a.xg[1][1])), 0.f);
            __syncthreads();
            if (gate_warp1) {
                float h = row_sum(OPS - 1) + gt[OPS - 1].bias;
                if (CELL == kR1GruRb) {
                    const float n = tanhf(h), hp = gt[0].on ? vr[gt[0].u] : 0.f;
                    h = (1.f - zg) * n + zg * hp;
                }
                if (more || layer + 1 < a.L) publish(0, OPS - 1, h, t);
                if (gt[OPS - 1].on && g == 0) {
                    if (layer == a.L - 1 && a.y) a.y[(size_t)t * S + gt[OPS - 1].u] = h;
                    if (!more && a.hT) a.hT[(size_t)layer * S + gt[OPS - 1].u] = h;
                }
            }
        }
        // ---- the next input: from the layer below (layer 0 has put it in place already)
        if (layer > 0 && more) {
            poll_take(wi, slot(0, below, t + 1), a.words[0][below], a.wmap[0][below], base + (uint32_t)(t + 1), vu);
            if (!__syncthreads_and(ok)) break;
        }
    }
    if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
}

// Everything one (cell, layer stack) needs on the device; built on first use and kept until one of
// its matrices is freed.
struct Rnn1Plan {
    int cell = 0, L = 0, device = 0, n_ctas = 0, H = 0, S = 0, val_dtype = 0;
    bool unusable = false;
    std::vector<uint64_t> uids;
    R1Args a{};
    size_t smem = 0;
    const void* kernel = nullptr;
    std::vector<void*> owned;                  // device memory
    uint32_t* h_status = nullptr;
    float* d_stage = nullptr; size_t stage_cap = 0;      // host I/O
    ~Rnn1Plan() {
        for (void* p : owned) cudaFree(p);
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

template <typename T>
static const void* pick_kernel(int cell) {
    switch (cell) {
        case kR1Lstm: return (const void*)csb_rnn1_kernel<T, kR1Lstm>;
        case kR1Gru: return (const void*)csb_rnn1_kernel<T, kR1Gru>;
        case kR1Lstmp: return (const void*)csb_rnn1_kernel<T, kR1Lstmp>;
        case kR1Ligru: return (const void*)csb_rnn1_kernel<T, kR1Ligru>;
        default: return (const void*)csb_rnn1_kernel<T, kR1GruRb>;
    }
}

static int env_int(const char* name, int dflt) {
    const char* v = getenv(name);
    return v && *v ? atoi(v) : dflt;
}

template <typename V>
static int put(Rnn1Plan* P, const V* h, size_t n, V** d) {
    const size_t bytes = std::max<size_t>(n, 1) * sizeof(V);
    CSB_CUDA(cudaMalloc((void**)d, bytes));
    P->owned.push_back(*d);
    if (h) { if (n) CSB_CUDA(cudaMemcpy(*d, h, n * sizeof(V), cudaMemcpyHostToDevice)); }
    else CSB_CUDA(cudaMemset(*d, 0, bytes));
    return CSB_OK;
}

// Returns 1 (and marks the plan) when the kernel does not take these matrices.
static int build_plan(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, Rnn1Plan* P) {
    const csb_matrix* A0 = W[0];
    P->cell = cell; P->L = L; P->device = A0->device; P->H = H; P->S = S; P->val_dtype = A0->val_dtype;
    P->unusable = true;
    for (int l = 0; l < L; ++l) P->uids.push_back(W[l]->uid);
    if (Wp) for (int l = 0; l < L; ++l) P->uids.push_back(Wp[l]->uid);
    int64_t weights = 0;
    for (int l = 0; l < L; ++l) {
        weights += W[l]->nnz + (Wp ? Wp[l]->nnz : 0);
        if (W[l]->val_dtype != A0->val_dtype || (Wp && Wp[l]->val_dtype != A0->val_dtype)) return 1;
    }
    int want = (int)std::min<int64_t>(A0->sm_count, std::max<int64_t>(L, weights / env_int("CSB_R1_MIN", 1024)));
    want = std::min(A0->sm_count, env_int("CSB_R1_CTAS", want));
    R1HostPlan Hp;
    const int hrc = plan_rnn1_host(cell, L, W, Wp, in_size, H, S, want, &Hp);
    if (hrc != CSB_OK) return hrc;
    R1Args& a = P->a;
    size_t at = Hp.max_smem;
    auto room = [&](size_t bytes) { const size_t o = at; at = (at + bytes + 15) & ~(size_t)15; return (uint32_t)o; };
    int max_in = 0;
    for (int l = 0; l < L; ++l) max_in = std::max(max_in, in_size[l]);
    // the gathered inputs of the input parts are used up before those of the recurrent part are written,
    // and those before the second product's: they share their room
    const size_t x00 = (Hp.max_xg[0][0] * 4 + 15) & ~(size_t)15;
    const uint32_t xg = room(std::max(std::max(x00 + Hp.max_xg[1][0] * 4, Hp.max_xg[0][1] * 4), Hp.max_xg[1][1] * 4));
    a.xg[0][0] = a.xg[0][1] = a.xg[1][1] = xg; a.xg[1][0] = xg + (uint32_t)x00;
    a.vu = room((size_t)(max_in + 1) * 4); a.vr = room((size_t)(S + 1) * 4); a.vm = room((size_t)(H + 1) * 4);
    a.part = room((size_t)kR1Threads * 8); a.misc = room(16);
    P->smem = at;
    if (P->smem > A0->smem_optin) return 1;
    P->n_ctas = (int)Hp.ctas.size();
    P->kernel = P->val_dtype == CSB_F16 ? pick_kernel<__half>(cell) : pick_kernel<float>(cell);
    CSB_CUDA(cudaFuncSetAttribute(P->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A0->smem_optin));
    int occ = 0;
    CSB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, P->kernel, kR1Threads, P->smem));
    if (occ < 1 || P->n_ctas > occ * A0->sm_count) return 1;     // the grid must be co-resident
    int rc;
    uint8_t* d_img = nullptr; R1Cta* d_ctas = nullptr;
    if ((rc = put(P, Hp.bytes.data(), Hp.bytes.size(), &d_img)) != CSB_OK || (rc = put(P, Hp.ctas.data(), Hp.ctas.size(), &d_ctas)) != CSB_OK) return rc;
    a.images = d_img; a.ctas = d_ctas;
    for (int e = 0; e < r1_ops(cell); ++e)
        for (int l = 0; l < L; ++l) {
            const std::vector<uint32_t>& m = Hp.wmap[e][l];
            uint32_t* d_map = nullptr;
            if ((rc = put(P, m.data(), m.size(), &d_map)) != CSB_OK) return rc;
            if ((rc = put(P, (const uint4*)nullptr, m.size() * kR1Ring, &a.ex[e][l])) != CSB_OK) return rc;
            a.wmap[e][l] = d_map; a.words[e][l] = (int)m.size();
        }
    if ((rc = put(P, (const uint32_t*)nullptr, (size_t)P->n_ctas, &a.epoch)) != CSB_OK || (rc = put(P, (const uint32_t*)nullptr, (size_t)kMaxLayers, &a.progress)) != CSB_OK) return rc;
    for (int l = 0; l < L; ++l) { a.in_size[l] = in_size[l]; a.layer_ctas[l] = Hp.layer_ctas[l]; }
    a.H = H; a.S = S; a.L = L;
    CSB_CUDA(cudaHostAlloc((void**)&P->h_status, 4, cudaHostAllocMapped));
    *P->h_status = 0;
    CSB_CUDA(cudaHostGetDevicePointer((void**)&a.status, P->h_status, 0));
    CSB_CUDA(cudaDeviceSynchronize());
    P->unusable = false;
    return CSB_OK;
}

int rnn1_forward(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const float* const* bias, const float* x, int64_t T,
                 int H, int S, const int* in_size, const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags, void* stream) {
    if (env_int("CSB_RNN_NO_RNN1", 0)) return 1;
    Rnn1Plan* P = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_r1_mu);
        for (auto& p : g_r1_plans) {
            if (p->cell != cell || p->L != L) continue;
            bool same = true;
            for (int l = 0; l < L; ++l) same = same && p->uids[l] == W[l]->uid && (!Wp || p->uids[L + l] == Wp[l]->uid);
            if (same) { P = p.get(); break; }
        }
        if (!P) {
            std::unique_ptr<Rnn1Plan> np(new Rnn1Plan());
            int rc;
            try { rc = build_plan(cell, L, W, Wp, in_size, H, S, np.get()); }
            catch (const std::bad_alloc&) { set_error("out of host memory while planning the time loop"); rc = CSB_ERR_ALLOC; }
            if (rc != CSB_OK && rc != 1) return rc;
            P = np.get();
            g_r1_plans.push_back(std::move(np));
        }
    }
    if (P->unusable) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const bool host_io = (flags & CSB_FLAG_HOST_IO) != 0, has_c = cell == kR1Lstm || cell == kR1Lstmp;
    const size_t nx = (size_t)T * in_size[0], ny = y ? (size_t)T * S : 0, nh = (size_t)L * S, nc = has_c ? (size_t)L * H : 0;
    R1Args a = P->a;
    a.x = x; a.h0 = h0; a.c0 = has_c ? c0 : nullptr; a.y = y; a.hT = hT; a.cT = has_c ? cT : nullptr;
    if (host_io) {
        const size_t need = nx + ny + 2 * nh + 2 * nc;
        if (need > P->stage_cap) {
            CSB_CUDA(cudaStreamSynchronize(st));
            cudaFree(P->d_stage); P->d_stage = nullptr; P->stage_cap = 0;
            CSB_CUDA(cudaMalloc((void**)&P->d_stage, need * 4));
            P->stage_cap = need;
        }
        float* d = P->d_stage;
        auto in = [&](const float*& p, size_t n) -> cudaError_t {
            if (!p) return cudaSuccess;
            const cudaError_t e = cudaMemcpyAsync(d, p, n * 4, cudaMemcpyHostToDevice, st);
            p = d; d += n;
            return e;
        };
        auto out = [&](float*& p, size_t n) { if (p) { p = d; d += n; } };
        CSB_CUDA(in(a.x, nx));
        CSB_CUDA(in(a.h0, nh));
        CSB_CUDA(in(a.c0, nc));
        out(a.y, ny); out(a.hT, nh); out(a.cT, nc);
    }
    for (int l = 0; l < L; ++l) a.bias[l] = bias ? bias[l] : nullptr;
    a.T = (int)T;
    uint32_t extra = 0;
    barrier_test_hook(&extra, &a.limit_ns);
    a.never = extra ? 0x40000000u : 0u;
    *P->h_status = 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)P->n_ctas); cfg.blockDim = dim3(kR1Threads); cfg.dynamicSmemBytes = P->smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    void* params[] = {(void*)&a};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, P->kernel, params);
    if (e == cudaErrorCooperativeLaunchTooLarge) { set_error("cooperative launch too large"); return CSB_ERR_LAUNCH; }
    CSB_CUDA(e);
    if (host_io) {
        if (y) CSB_CUDA(cudaMemcpyAsync(y, a.y, ny * 4, cudaMemcpyDeviceToHost, st));
        if (hT) CSB_CUDA(cudaMemcpyAsync(hT, a.hT, nh * 4, cudaMemcpyDeviceToHost, st));
        if (has_c && cT) CSB_CUDA(cudaMemcpyAsync(cT, a.cT, nc * 4, cudaMemcpyDeviceToHost, st));
    }
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
