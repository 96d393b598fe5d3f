// Resident time loop of the recurrent cells (LSTM, GRU, LSTMP, Li-GRU, reset-before GRU) for small
// batches: one cooperative launch per sequence (Section 2.1 of the paper: per step a CSB product with
// [u_t ; h_{t-1}], then the element-wise gate arithmetic, the c / h "context link" feeding the next step).
//
// A CTA owns a range of hidden units of one layer (csb_rnn1.hpp); its weights stay in shared memory.
// What bounds a step is latency: the exchange of h_t between CTAs, then product, sums and gates, and
// inside the product the traffic of shared memory.  So
//   * a vector crosses CTAs as 16-byte words of three values and the number of their step, written
//     and read with single 16-byte accesses (relaxed, 128-bit atomic): a reader that sees the step
//     it waits for also holds the values.  No fence, no counter, no grid barrier; layers run as a
//     dataflow pipeline.  Step numbers go on from call to call (a word per CTA keeps the count), so
//     nothing is cleared between calls.  A vector stays for 32 steps; every 8 steps a layer checks
//     that the layer above has read what it is about to overwrite;
//   * the product over the input part [u_t] is done while h_{t-1} is on its way, and u_{t+1} is fetched
//     into the other of two buffers meanwhile;
//   * a lane of the product fetches up to 8 inputs through the column indices into registers and
//     multiplies them with the rows of its task one after the other; partial sums go to places of
//     their own, ordered by row.  Measured at 2 x 2048 units, 10x pruned, batch 1: FIXME_WALK
//   * three barriers a step: inputs complete, partial sums complete, row sums complete.
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
    const uint32_t* wmap[2][kMaxLayers];       // first element | elements << 24 of every exchange word
    int words[2][kMaxLayers];
    uint4* ex[2][kMaxLayers];                  // [kR1Ring][words]
    uint32_t* epoch;                           // per CTA: step numbers used so far
    uint32_t* progress;                        // per layer: blocks of kR1Block input steps read, summed over its CTAs, never cleared
    int layer_ctas[kMaxLayers];
    uint32_t* status;
    unsigned long long limit_ns;
    uint32_t never;                            // test hook: wait for step numbers that never come
    int T, B, H, S, L;
    uint32_t vu[2], vr, vm, part[2], z[2], cs, bias0, bias1, misc;   // shared-memory offsets behind the image
#ifdef CSB_PHASE_CLOCKS
    long long* clocks;                         // [CTA][8] cycles of thread 0 summed over the steps
#endif
};
#ifdef CSB_PHASE_CLOCKS
#define R1_LAP(i) do { if (tid == 0) { const long long n_ = clock64(); lap[i] += n_ - lap_at; lap_at = n_; } } while (0)
#else
#define R1_LAP(i) do { } while (0)
#endif

typedef unsigned __int128 Word;                // three values and a step number
__device__ __forceinline__ Word ld_word(const uint4* p) {
    Word w;
    asm volatile("ld.relaxed.gpu.global.b128 %0, [%1];" : "=q"(w) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ void st_word(uint4* p, float a, float b, float c, uint32_t tag) {
    const Word w = (Word)__float_as_uint(a) | ((Word)__float_as_uint(b) << 32) | ((Word)__float_as_uint(c) << 64) | ((Word)tag << 96);
    asm volatile("st.relaxed.gpu.global.b128 [%0], %1;" ::"l"(p), "q"(w) : "memory");
}
__device__ __forceinline__ uint32_t word_tag(Word w) { return (uint32_t)(w >> 96); }
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)), "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 half2_to_float2(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }
__device__ __forceinline__ float logistic(float a) { return 1.f / (1.f + expf(-a)); }

// N consecutive 32-bit words of shared memory.
template <int N> struct Regs { uint32_t v[N]; };
template <int N>
__device__ __forceinline__ Regs<N> ld_regs(const uint8_t* p) {
    Regs<N> r;
    if (N == 1) r.v[0] = *reinterpret_cast<const uint32_t*>(p);
    if (N == 2) { const uint2 t = *reinterpret_cast<const uint2*>(p); r.v[0] = t.x; r.v[N > 1 ? 1 : 0] = t.y; }
#pragma unroll
    for (int i = 0; i + 4 <= N; i += 4) {
        const uint4 t = *reinterpret_cast<const uint4*>(p + 4 * i);
        r.v[i] = t.x; r.v[i + 1 < N ? i + 1 : 0] = t.y; r.v[i + 2 < N ? i + 2 : 0] = t.z; r.v[i + 3 < N ? i + 3 : 0] = t.w;
    }
    return r;
}

// One group of tasks with K columns: inputs into registers, then row after row.
template <typename T, int BT, int K>
__device__ __forceinline__ void walk_group(const uint8_t* img, const R1Group& g, int lane, const float* v, float* partials) {
    constexpr int kWords = K * (int)sizeof(T) / 4;         // weight words of a row
    const Regs<K / 2> c = ld_regs<K / 2>(img + g.cols_off + lane * (K * 2));
    float x[K][BT];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float* p = v + (size_t)((c.v[k / 2] >> (16 * (k & 1))) & 0xffffu) * BT;
        if (BT == 1) x[k][0] = *p;
        if (BT == 2) { const float2 t = *reinterpret_cast<const float2*>(p); x[k][0] = t.x; x[k][BT > 1 ? 1 : 0] = t.y; }
#pragma unroll
        for (int b = 0; b + 4 <= BT; b += 4) {
            const float4 t = *reinterpret_cast<const float4*>(p + b);
            x[k][b] = t.x; x[k][b + 1 < BT ? b + 1 : 0] = t.y; x[k][b + 2 < BT ? b + 2 : 0] = t.z; x[k][b + 3 < BT ? b + 3 : 0] = t.w;
        }
    }
    const uint8_t* w = img + g.w_off + lane * (kWords == 8 ? 16 : kWords * 4);
    const uint32_t* pos = reinterpret_cast<const uint32_t*>(img + g.pos_off) + lane;
    auto row = [&](const Regs<kWords>& q, uint32_t place) {
        float wf[K];
#pragma unroll
        for (int i = 0; i < kWords; ++i) {
            if (sizeof(T) == 2) { const float2 t = half2_to_float2(q.v[i]); wf[(2 * i) % K] = t.x; wf[(2 * i + 1) % K] = t.y; }
            else wf[i % K] = __uint_as_float(q.v[i]);
        }
        float* out = partials + place * BT;
        if (BT == 1) {
            float2 a = make_float2(wf[0] * x[0][0], wf[1] * x[1][0]);
#pragma unroll
            for (int k = 2; k < K; k += 2) a = fma2(make_float2(wf[k], wf[k + 1]), make_float2(x[k][0], x[k + 1][0]), a);
            *out = a.x + a.y;
        } else {
            float2 a[BT / 2 > 0 ? BT / 2 : 1];
#pragma unroll
            for (int b = 0; b < BT / 2; ++b) a[b] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k)
#pragma unroll
                for (int b = 0; b < BT / 2; ++b) a[b] = fma2(make_float2(wf[k], wf[k]), make_float2(x[k][2 * b], x[k][(2 * b + 1) % BT]), a[b]);
            if (BT == 2) *reinterpret_cast<float2*>(out) = a[0];
#pragma unroll
            for (int b = 0; b + 1 < BT / 2; b += 2)
                *reinterpret_cast<float4*>(out + 2 * b) = make_float4(a[b].x, a[b].y, a[(b + 1) % (BT / 2 > 0 ? BT / 2 : 1)].x, a[(b + 1) % (BT / 2 > 0 ? BT / 2 : 1)].y);
        }
    };
    auto load = [&](int r) {
        if (kWords == 8) {                                 // fp32, eight columns: [half][lane]
            const Regs<4> lo = ld_regs<4>(w + (size_t)r * 1024), hi = ld_regs<4>(w + (size_t)r * 1024 + 512);
            Regs<kWords> q;
#pragma unroll
            for (int i = 0; i < 4; ++i) { q.v[i % kWords] = lo.v[i]; q.v[(4 + i) % kWords] = hi.v[i]; }
            return q;
        }
        return ld_regs<kWords>(w + (size_t)r * (32 * kWords * 4));
    };
    int r = 0;
    for (; r + 2 <= g.rows; r += 2) {
        const uint32_t p = pos[(r / 2) * 32];
        const Regs<kWords> a = load(r), b = load(r + 1);
        row(a, p & 0xffffu);
        row(b, p >> 16);
    }
    if (r < g.rows) row(load(r), pos[(r / 2) * 32] & 0xffffu);
}

// A warp's groups [g0, g0 + n) of one product.
template <typename T, int BT>
__device__ __forceinline__ void walk(const uint8_t* img, const R1Group* groups, int n, int lane, const float* v, float* partials) {
    constexpr int kWide = BT >= 8 ? 4 : 8;                 // r1_wide()
    for (int i = 0; i < n; ++i) {
        const R1Group g = groups[i];
        if (g.narrow) walk_group<T, BT, kWide / 2>(img, g, lane, v, partials);
        else walk_group<T, BT, kWide>(img, g, lane, v, partials);
    }
}

template <typename T, int CELL, int BT>
__global__ void __launch_bounds__(kR1Threads, 1) csb_rnn1_kernel(const __grid_constant__ R1Args a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int OPS = CELL == kR1Lstmp || CELL == kR1GruRb ? 2 : 1;
    constexpr int G0 = CELL == kR1Lstm || CELL == kR1Lstmp ? 4 : CELL == kR1Gru ? 3 : 2;
    constexpr bool kHasC = CELL == kR1Lstm || CELL == kR1Lstmp;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const R1Cta me = a.ctas[blockIdx.x];
    const int layer = me.layer, below = layer - 1, I = a.in_size[layer], S = a.S, H = a.H, T_ = a.T, B = a.B;
    const uint8_t* img = smem;
    auto f32 = [&](uint32_t off) { return reinterpret_cast<float*>(smem + off); };
    float* vr = f32(a.vr);
    float* vm = f32(a.vm);
    float* cs = f32(a.cs);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + a.misc);
    volatile int* s_ok = reinterpret_cast<volatile int*>(smem + a.misc + 8);

    // ---- weights; initial state; first input.  A staged vector holds BT values per column and ends in zeros.
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
        mbar_expect_tx(bar, me.bytes);
        const uint8_t* src = a.images + (size_t)me.off16 * 16;
        for (uint32_t off = 0; off < me.bytes; off += 16384u) bulk_g2s(smem + off, src + off, min(16384u, me.bytes - off), bar);
        *s_ok = 1;
    }
    auto stage = [&](float* dst, const float* src, int n) {      // [B][n] in global memory
        for (int b = 0; b < BT; ++b)
            for (int i = tid; i < n; i += kR1Threads) dst[i * BT + b] = src && b < B ? __ldg(src + (size_t)b * n + i) : 0.f;
    };
    stage(vr, a.h0 ? a.h0 + (size_t)layer * B * S : nullptr, S);
    if (layer == 0) stage(f32(a.vu[0]), a.x, I);
    if (tid < BT) { vr[S * BT + tid] = 0.f; f32(a.vu[0])[I * BT + tid] = 0.f; f32(a.vu[1])[I * BT + tid] = 0.f; if (OPS == 2) vm[H * BT + tid] = 0.f; }
    if (layer == 0 && BT > 1)                                    // batch columns past B stay zero
        for (int i = tid; i < I * BT; i += kR1Threads) if (i % BT >= B) f32(a.vu[1])[i] = 0.f;
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
    const R1Header* hd = reinterpret_cast<const R1Header*>(img);
    const int U0 = hd->op[0].units, U1 = OPS == 2 ? hd->op[OPS - 1].units : 0;
    // places of partial sums that no task writes stay zero; cell state and bias of the CTA's units
#pragma unroll
    for (int op = 0; op < OPS; ++op) for (int i = tid; i < (int)hd->op[op].partials * BT; i += kR1Threads) f32(a.part[op])[i] = 0.f;
    if (kHasC)
        for (int i = tid; i < U0 * BT; i += kR1Threads) {
            const int u = i / BT, b = i % BT;
            cs[i] = a.c0 && b < B ? __ldg(a.c0 + ((size_t)layer * B + b) * H + hd->op[0].unit0 + u) : 0.f;
        }
    const float* bl = a.bias[layer];
    for (int i = tid; i < 4 * U0; i += kR1Threads) {
        const int g = i / U0, u = i % U0;
        f32(a.bias0)[i] = bl && g < (CELL == kR1Gru ? 4 : G0) ? __ldg(bl + (size_t)g * H + hd->op[0].unit0 + u) : 0.f;
    }
    if (OPS == 2)
        for (int u = tid; u < U1; u += kR1Threads) f32(a.bias1)[u] = bl && CELL == kR1GruRb ? __ldg(bl + (size_t)2 * H + hd->op[OPS - 1].unit0 + u) : 0.f;
    struct Walk { const R1Group* g; int n[2]; } wk[OPS];
#pragma unroll
    for (int op = 0; op < OPS; ++op) {
        const uint16_t* wd = reinterpret_cast<const uint16_t*>(img + hd->op[op].warp_off) + warp * 4;
        wk[op].g = reinterpret_cast<const R1Group*>(img + hd->op[op].groups_off) + wd[0];
        wk[op].n[0] = wd[1]; wk[op].n[1] = wd[2];
    }
    // row sums: 2^lp neighbouring lanes per row
    int lp[OPS];
#pragma unroll
    for (int op = 0; op < OPS; ++op) { lp[op] = 0; while (lp[op] < 5 && (hd->op[op].n_rows << (lp[op] + 1)) <= kR1Threads) ++lp[op]; }

    // ---- the exchange.  The first words are asked for early (poll_issue), all are taken in poll_take.
    uint4* ex_state = a.ex[0][layer];
    const int n_state = a.words[0][layer];
    const uint32_t* map_state = a.wmap[0][layer];
    uint4* ex_mid = OPS == 2 ? a.ex[1][layer] : nullptr;
    const int n_mid = OPS == 2 ? a.words[1][layer] : 0;
    const uint32_t* map_mid = OPS == 2 ? a.wmap[1][layer] : nullptr;
    const uint4* ex_below = layer > 0 ? a.ex[0][below] : nullptr;
    const int n_below = layer > 0 ? a.words[0][below] : 0;
    const uint32_t* map_below = layer > 0 ? a.wmap[0][below] : nullptr;
    auto poll_issue = [&](Word (&w)[kR1Words], const uint4* src, int n) {
#pragma unroll
        for (int q = 0; q < kR1Words; ++q) if (tid + q * kR1Threads < n) w[q] = ld_word(src + tid + q * kR1Threads);
    };
    auto take_word = [&](Word w, const uint4* src, const uint32_t* map, int i, uint32_t want, float* dst) {
        unsigned long long t0 = 0;
        unsigned int spins = 0;
        while (word_tag(w) != want) {
            if (*s_ok == 0) { ok = false; break; }         // another thread has given up
            if ((++spins & 63u) == 0) {
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                else if (now - t0 > a.limit_ns) { *(volatile uint32_t*)a.status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; ok = false; break; }
            }
            w = ld_word(src + i);
        }
        const uint32_t m = __ldg(map + i);
        float* p = dst + (m & 0xffffffu);
        p[0] = __uint_as_float((uint32_t)w);
        if ((m >> 24) > 1) p[1] = __uint_as_float((uint32_t)(w >> 32));
        if ((m >> 24) > 2) p[2] = __uint_as_float((uint32_t)(w >> 64));
    };
    auto poll_take = [&](Word (&w)[kR1Words], const uint4* src, int n, const uint32_t* map, uint32_t want, float* dst) {
        want += a.never;
#pragma unroll
        for (int q = 0; q < kR1Words; ++q) if (tid + q * kR1Threads < n) take_word(w[q], src, map, tid + q * kR1Threads, want, dst);
        for (int i = tid + kR1Words * kR1Threads; i < n; i += kR1Threads) take_word(ld_word(src + i), src, map, i, want, dst);
    };
    // The sums of a product's rows over their partial sums (GRU: input and recurrent part apart).
    auto row_sums = [&](int op) {
        const R1Row* rows = reinterpret_cast<const R1Row*>(img + hd->op[op].rows_off);
        const float* P = f32(a.part[op]);
        float* z = f32(a.z[op]);
        const int n = hd->op[op].n_rows, lanes = 1 << lp[op], s = tid & (lanes - 1);
        for (int r0 = 0; r0 < n; r0 += kR1Threads >> lp[op]) {
            const int r = r0 + (tid >> lp[op]);
            float sum[2][BT];
#pragma unroll
            for (int b = 0; b < BT; ++b) { sum[0][b] = 0.f; sum[1][b] = 0.f; }
            if (r < n) {
                const R1Row d = rows[r];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const float* q = P + (size_t)d.base[p] * 4 * BT;
                    for (int i = s; i < d.quads[p]; i += lanes)
#pragma unroll
                        for (int k = 0; k < BT; ++k) {     // BT float4: four places of BT values
                            const float4 t = *reinterpret_cast<const float4*>(q + ((size_t)i * BT + k) * 4);
                            const float e[4] = {t.x, t.y, t.z, t.w};
                            float* acc = sum[CELL == kR1Gru ? p : 0];
                            if (BT == 1) acc[0] += (e[0] + e[1]) + (e[2] + e[3]);
                            else
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[(4 * k + j) % BT] += e[j];
                        }
                }
            }
            for (int off = lanes >> 1; off >= 1; off >>= 1)
#pragma unroll
                for (int b = 0; b < BT; ++b) {
                    sum[0][b] += __shfl_xor_sync(0xffffffffu, sum[0][b], off);
                    if (CELL == kR1Gru) sum[1][b] += __shfl_xor_sync(0xffffffffu, sum[1][b], off);
                }
            if (r < n && s == 0)
#pragma unroll
                for (int b = 0; b < BT; ++b) {
                    if (CELL == kR1Gru) {
                        const bool cand = r >= 2 * U0;     // the candidate's two parts stay apart: slots 2 and 3
                        z[r * BT + b] = cand ? sum[0][b] : sum[0][b] + sum[1][b];
                        if (cand) z[(r + U0) * BT + b] = sum[1][b];
                    } else z[r * BT + b] = sum[0][b];
                }
        }
    };
    Word wr[kR1Words] = {}, wi[kR1Words] = {};
    if (layer > 0) {
        poll_issue(wi, ex_below, n_below);
        poll_take(wi, ex_below, n_below, map_below, base, f32(a.vu[0]));
    }
    if (!__syncthreads_and(ok)) {
        if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
        return;
    }
#ifdef CSB_PHASE_CLOCKS
    long long lap[8] = {0, 0, 0, 0, 0, 0, 0, 0}, lap_at = clock64();
#endif
    const int j = lane >> 2, g = lane & 3;                 // gate lanes: four per state, six states per warp and round
    for (int t = 0; t < T_; ++t) {
        const bool more = t + 1 < T_;
        const float* vu = f32(a.vu[t & 1]);
        float* vu_next = f32(a.vu[(t + 1) & 1]);
        // ---- u_t lies in vu: its part of the product, while h_{t-1} and u_{t+1} are on their way
        const uint4* rec_src = ex_state + (size_t)((t - 1) & (kR1Ring - 1)) * n_state;
        const uint4* next_src = ex_below + (size_t)((t + 1) & (kR1Ring - 1)) * n_below;
        if (layer == 0 && more)
            for (int b = 0; b < B; ++b)
                for (int i = tid; i < I; i += kR1Threads) cp_async4(vu_next + i * BT + b, a.x + ((size_t)(t + 1) * B + b) * I + i);
        if (t > 0) poll_issue(wr, rec_src, n_state);
        walk<T, BT>(img, wk[0].g, wk[0].n[0], lane, vu, f32(a.part[0]));
        if (CELL == kR1GruRb) walk<T, BT>(img, wk[OPS - 1].g, wk[OPS - 1].n[0], lane, vu, f32(a.part[1]));
        R1_LAP(0);                                         // product of the input part
        if (t > 0) poll_take(wr, rec_src, n_state, map_state, base + (uint32_t)(t - 1), vr);
        if (layer > 0 && more) poll_issue(wi, next_src, n_below);
        R1_LAP(1);                                         // the state of the step before
        if (!__syncthreads_and(ok)) break;
        R1_LAP(2);
        if (layer > 0 && tid == 0 && (t & (kR1Block - 1)) == kR1Block - 1) atomicAdd(a.progress + layer, 1u);   // u up to step t has been read
        walk<T, BT>(img, wk[0].g + wk[0].n[0], wk[0].n[1], lane, vr, f32(a.part[0]));
        R1_LAP(3);                                         // product of the recurrent part
        if (layer > 0 && more) poll_take(wi, next_src, n_below, map_below, base + (uint32_t)(t + 1), vu_next);
        if (layer == 0 && more) cp_async_wait();
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
        row_sums(0);
        __syncthreads();
        R1_LAP(4);                                         // row sums
        // ---- gates: lane g of a state's four applies gate g
        const int E0 = U0 * BT;
        for (int e0 = warp * kR1WarpUnits; e0 < E0; e0 += kR1Warps * kR1WarpUnits) {
            const int e = e0 + j, l0 = lane & ~3;
            const bool on = j < kR1WarpUnits && e < E0;
            const int u = on ? e / BT : 0, b = on ? e % BT : 0;
            float z = on && g < (CELL == kR1Gru ? 4 : G0) ? f32(a.z[0])[g * E0 + e] + f32(a.bias0)[g * U0 + u] : 0.f;
            const int at = ((int)hd->op[0].unit0 + u) * BT + b;      // the state's element in the staged vectors
            const float hp = CELL == kR1Gru || CELL == kR1Ligru || CELL == kR1GruRb ? vr[at] : 0.f;
            float h, c = 0.f;
            if (kHasC) {
                c = on ? cs[e] : 0.f;
                z = g == 2 ? tanhf(z) : logistic(z);
                const float zi = __shfl_sync(0xffffffffu, z, l0), zf = __shfl_sync(0xffffffffu, z, l0 + 1);
                const float zc = __shfl_sync(0xffffffffu, z, l0 + 2), zo = __shfl_sync(0xffffffffu, z, l0 + 3);
                c = zf * c + zi * zc;
                h = zo * tanhf(c);
                if (on && g == 0) cs[e] = c;
            } else if (CELL == kR1Gru) {
                if (g < 2) z = logistic(z);
                const float r = __shfl_sync(0xffffffffu, z, l0), zz = __shfl_sync(0xffffffffu, z, l0 + 1);
                const float ni = __shfl_sync(0xffffffffu, z, l0 + 2), nh = __shfl_sync(0xffffffffu, z, l0 + 3);
                h = (1.f - zz) * tanhf(ni + r * nh) + zz * hp;
            } else if (CELL == kR1Ligru) {
                if (g == 0) z = logistic(z);
                const float zz = __shfl_sync(0xffffffffu, z, l0), cand = fmaxf(__shfl_sync(0xffffffffu, z, l0 + 1), 0.f);
                h = zz * hp + (1.f - zz) * cand;
            } else {
                z = logistic(z);
                if (on && g == 1) cs[e] = z;               // the update gate, for the second half of the step
                h = __shfl_sync(0xffffffffu, z, l0) * hp;  // r * h_{t-1}
            }
            const float h1 = __shfl_down_sync(0xffffffffu, h, 4), h2 = __shfl_down_sync(0xffffffffu, h, 8);
            uint4* ex = OPS == 2 ? ex_mid + (size_t)(t & (kR1Ring - 1)) * n_mid : ex_state + (size_t)(t & (kR1Ring - 1)) * n_state;
            if (on && g == 0 && (j == 0 || j == 3) && (OPS == 2 || more || layer + 1 < a.L)) st_word(ex + hd->op[0].word0 + e / 3, h, h1, h2, base + (uint32_t)t);
            if (on && g == 0 && b < B) {
                if (OPS == 1) {
                    if (layer == a.L - 1 && a.y) a.y[((size_t)t * B + b) * S + at / BT] = h;
                    if (!more && a.hT) a.hT[((size_t)layer * B + b) * S + at / BT] = h;
                }
                if (kHasC && !more && a.cT) a.cT[((size_t)layer * B + b) * H + at / BT] = c;
            }
        }
        R1_LAP(5);                                         // gates
        if (OPS == 2) {
            // ---- second product of the step: what the first one gave, from every CTA of the layer
            const uint4* src = ex_mid + (size_t)(t & (kR1Ring - 1)) * n_mid;
            poll_issue(wr, src, n_mid);
            poll_take(wr, src, n_mid, map_mid, base + (uint32_t)t, vm);
            if (!__syncthreads_and(ok)) break;
            R1_LAP(6);                                     // exchange inside the step
            walk<T, BT>(img, wk[OPS - 1].g + wk[OPS - 1].n[0], wk[OPS - 1].n[1], lane, vm, f32(a.part[1]));
            __syncthreads();
            row_sums(OPS - 1);
            __syncthreads();
            const int E1 = U1 * BT;
            for (int e0 = warp * kR1WarpUnits; e0 < E1; e0 += kR1Warps * kR1WarpUnits) {
                const int e = e0 + j;
                const bool on = j < kR1WarpUnits && e < E1;
                const int u = on ? e / BT : 0, b = on ? e % BT : 0, at = ((int)hd->op[OPS - 1].unit0 + u) * BT + b;
                float h = on ? f32(a.z[1])[e] + f32(a.bias1)[u] : 0.f;
                if (CELL == kR1GruRb && on) { const float zz = cs[e]; h = (1.f - zz) * tanhf(h) + zz * vr[at]; }
                const float h1 = __shfl_down_sync(0xffffffffu, h, 4), h2 = __shfl_down_sync(0xffffffffu, h, 8);
                if (on && g == 0 && (j == 0 || j == 3) && (more || layer + 1 < a.L))
                    st_word(ex_state + (size_t)(t & (kR1Ring - 1)) * n_state + hd->op[OPS - 1].word0 + e / 3, h, h1, h2, base + (uint32_t)t);
                if (on && g == 0 && b < B) {
                    if (layer == a.L - 1 && a.y) a.y[((size_t)t * B + b) * S + at / BT] = h;
                    if (!more && a.hT) a.hT[((size_t)layer * B + b) * S + at / BT] = h;
                }
            }
            R1_LAP(7);                                     // second product, its sums and gates
        }
    }
#ifdef CSB_PHASE_CLOCKS
    if (tid == 0) for (int i = 0; i < 8; ++i) a.clocks[(size_t)blockIdx.x * 8 + i] = lap[i];
#endif
    if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
}

#ifdef CSB_PHASE_CLOCKS
static long long* g_r1_clocks = nullptr;
static int g_r1_clock_ctas = 0;
extern "C" int csb_debug_rnn1_clocks(long long* host_out, int max_ctas) {
    cudaMemcpy(host_out, g_r1_clocks, (size_t)std::min(max_ctas, g_r1_clock_ctas) * 8 * 8, cudaMemcpyDeviceToHost);
    return g_r1_clock_ctas;
}
#endif

// Everything one (cell, layer stack) needs on the device; built on first use and kept until one of
// its matrices is freed.
struct Rnn1Plan {
    int cell = 0, L = 0, BT = 1, device = 0, n_ctas = 0, H = 0, S = 0, val_dtype = 0;
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

template <typename T, int BT>
static const void* pick_kernel(int cell) {
    switch (cell) {
        case kR1Lstm: return (const void*)csb_rnn1_kernel<T, kR1Lstm, BT>;
        case kR1Gru: return (const void*)csb_rnn1_kernel<T, kR1Gru, BT>;
        case kR1Lstmp: return (const void*)csb_rnn1_kernel<T, kR1Lstmp, BT>;
        case kR1Ligru: return (const void*)csb_rnn1_kernel<T, kR1Ligru, BT>;
        default: return (const void*)csb_rnn1_kernel<T, kR1GruRb, BT>;
    }
}
template <typename T>
static const void* pick_kernel_bt(int cell, int BT) {
    return BT == 1 ? pick_kernel<T, 1>(cell) : nullptr;
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
static int build_plan(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, Rnn1Plan* P) {
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
    int want = (int)std::min<int64_t>(A0->sm_count, std::max<int64_t>(L, weights / env_int("CSB_R1_MIN", 1024)));
    want = std::min(A0->sm_count, env_int("CSB_R1_CTAS", want));
    R1HostPlan Hp;
    const int hrc = plan_rnn1_host(cell, L, W, Wp, in_size, H, S, BT, want, &Hp);
    if (hrc != CSB_OK) return hrc;
    R1Args& a = P->a;
    size_t at = Hp.max_bytes;
    auto room = [&](size_t floats) { const size_t o = at; at = (at + floats * 4 + 15) & ~(size_t)15; return (uint32_t)o; };
    int max_in = 0;
    for (int l = 0; l < L; ++l) max_in = std::max(max_in, in_size[l]);
    for (uint32_t& v : a.vu) v = room((size_t)(max_in + 1) * BT);
    a.vr = room((size_t)(S + 1) * BT); a.vm = room(r1_ops(cell) == 2 ? (size_t)(H + 1) * BT : 0);
    for (int op = 0; op < 2; ++op) a.part[op] = room(Hp.max_partials[op] * BT);
    a.z[0] = room(4 * Hp.max_units * BT); a.z[1] = room(r1_ops(cell) == 2 ? Hp.max_units * BT : 0);
    a.cs = room(Hp.max_units * BT); a.bias0 = room(4 * Hp.max_units); a.bias1 = room(Hp.max_units);
    a.misc = room(4);
    P->smem = at;
    if (P->smem > A0->smem_optin) return 1;
    P->n_ctas = (int)Hp.ctas.size();
    P->kernel = P->val_dtype == CSB_F16 ? pick_kernel_bt<__half>(cell, BT) : pick_kernel_bt<float>(cell, BT);
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

int rnn1_forward(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const float* const* bias, const float* x, int64_t T, int B,
                 int H, int S, const int* in_size, const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags, void* stream) {
    if (env_int("CSB_RNN_NO_RNN1", 0)) return 1;
    if (B > 1) return 1;
    const int BT = 1;
    Rnn1Plan* P = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_r1_mu);
        for (auto& p : g_r1_plans) {
            if (p->cell != cell || p->L != L || p->BT != BT) continue;
            bool same = true;
            for (int l = 0; l < L; ++l) same = same && p->uids[l] == W[l]->uid && (!Wp || p->uids[L + l] == Wp[l]->uid);
            if (same) { P = p.get(); break; }
        }
        if (!P) {
            std::unique_ptr<Rnn1Plan> np(new Rnn1Plan());
            int rc;
            try { rc = build_plan(cell, L, W, Wp, in_size, H, S, BT, np.get()); }
            catch (const std::bad_alloc&) { set_error("out of host memory while planning the time loop"); rc = CSB_ERR_ALLOC; }
            if (rc != CSB_OK && rc != 1) return rc;
            P = np.get();
            g_r1_plans.push_back(std::move(np));
        }
    }
    if (P->unusable) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const bool host_io = (flags & CSB_FLAG_HOST_IO) != 0, has_c = cell == kR1Lstm || cell == kR1Lstmp;
    const size_t nx = (size_t)T * B * in_size[0], ny = y ? (size_t)T * B * S : 0, nh = (size_t)L * B * S, nc = has_c ? (size_t)L * B * H : 0;
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
