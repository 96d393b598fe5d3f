// Resident time loop of the recurrent cells for small products (layout and reasons: csb_rnn_unit.hpp).
//
// As in csb_rnn1_kernel.cuh one cooperative launch runs the whole sequence and vectors cross CTAs as values
// that carry the number of their step; here every value has its own (8 bytes, written with one store;
// a reader takes two with one 16-byte load), because a warp publishes its units by itself.  A step of a
// warp: input part of its rows (while h_{t-1} is on its way), words of h_{t-1}, barrier, recurrent part,
// sums by shuffle, gates, publication.  Staged vectors are double-buffered, so that the one barrier is
// enough.
//
// What bounds it is the exchange: 0.9 to 1.0 us of a step of 1.9 (1024 LSTM units on 153 inputs, 13x
// pruned, 64 CTAs; 3.7 us with the other loop, whose sums and gates are phases of their own), the walks
// take 0.5 and sums and gates 0.4.  Words are asked for as late as they can be: a load that finds a pair not
// yet written has to be repeated, and many CTAs repeating theirs slow down the arrival itself.  With the
// loads in front of the input part the same step took 2.8 us.  So nothing is asked for before the input
// part is done, and pauses stand where a wait is sure to be long: the second exchange of a step (LSTMP 4.6 us
// without, 3.0 with 200 to 400 ns), and the state of stacked layers, of which two CTA sets read one
// (2 x 1024 units: 3.6 us without, 2.5 with 150 to 300 ns; a single layer has nothing to gain).  Pauses that
// adapt themselves, from hits and misses of the first load, did no better (3.3 and 2.5 us).
// The two constants fit 1024 units (us a step without / with them, batch 1, 10x pruned: two LSTM layers 3.88 / 2.54,
// LSTMP 4.77 / 3.07, reset-before GRU 3.95 / 3.06).  Small stacks, whose exchange is shorter, would do without: two LSTM
// layers of 256 units 2.01 / 2.16, LSTMP with 128 2.43 / 2.64, two reset-before layers of 64 2.66 / 3.06.
#pragma once

#include "csb_rnn_exchange.cuh"
#include "csb_rnn1_args.hpp"

namespace csb {

constexpr unsigned kStatePause = 150, kMidPause = 300;     // ns, see above

// s[b] += f * x[b]
template <int BT>
__device__ __forceinline__ void mul_add(const float* x, float f, float (&s)[BT]) {
    if (BT == 1) s[0] = fmaf(f, *x, s[0]);
#pragma unroll
    for (int b = 0; b + 4 <= BT; b += 4) {
        const float4 v = *reinterpret_cast<const float4*>(x + b);
        const float2 lo = fma2(make_float2(f, f), make_float2(v.x, v.y), make_float2(s[b], s[(b + 1) % BT]));
        const float2 hi = fma2(make_float2(f, f), make_float2(v.z, v.w), make_float2(s[(b + 2) % BT], s[(b + 3) % BT]));
        s[b] = lo.x; s[(b + 1) % BT] = lo.y; s[(b + 2) % BT] = hi.x; s[(b + 3) % BT] = hi.y;
    }
}

// A lane's pairs of one part.
template <typename T, int BT> struct UnitWalk;
template <int BT> struct UnitWalk<__half, BT> {
    static __device__ __forceinline__ void run(const uint8_t* list, int n, const float* v, float (&acc)[BT]) {
        const uint4* p = reinterpret_cast<const uint4*>(list);
        float alt[BT];
#pragma unroll
        for (int b = 0; b < BT; ++b) alt[b] = 0.f;
        auto pair = [&](uint32_t w, float (&s)[BT]) {
            mul_add<BT>(v + (size_t)(w & 0xffffu) * BT, __half2float(__ushort_as_half((unsigned short)(w >> 16))), s);
        };
#pragma unroll 2
        for (int i = 0; i < n; ++i, p += 32) {
            const uint4 w = *p;
            pair(w.x, acc);
            pair(w.y, alt);
            pair(w.z, acc);
            pair(w.w, alt);
        }
#pragma unroll
        for (int b = 0; b < BT; ++b) acc[b] += alt[b];
    }
};
template <int BT> struct UnitWalk<float, BT> {
    static __device__ __forceinline__ void run(const uint8_t* list, int n, const float* v, float (&acc)[BT]) {
        const uint4* p = reinterpret_cast<const uint4*>(list);
#pragma unroll 2
        for (int i = 0; i < n; ++i, p += 32) {
            const uint4 w = *p;
            mul_add<BT>(v + (size_t)w.x * BT, __uint_as_float(w.y), acc);
            mul_add<BT>(v + (size_t)w.z * BT, __uint_as_float(w.w), acc);
        }
    }
};

template <typename T, int CELL, int BT>
__global__ void __launch_bounds__(kR1Threads, 1) csb_rnn_unit_kernel(const __grid_constant__ RuArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int OPS = CELL == kR1Lstmp || CELL == kR1GruRb ? 2 : 1;
    constexpr int R0 = CELL == kR1Ligru || CELL == kR1GruRb ? 2 : 4;       // ru_rows()
    constexpr bool kHasC = CELL == kR1Lstm || CELL == kR1Lstmp;
    constexpr int kBtLog = BT == 1 ? 0 : BT == 4 ? 2 : 3;
    constexpr int kW = BT == 1 ? 2 : 4;                    // 16-byte loads of words a thread has under way
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const RuCta me = a.ctas[blockIdx.x];
    const int layer = me.layer, below = layer - 1, I = a.in_size[layer], S = a.S, H = a.H, T_ = a.T, B = a.B;
    auto f32 = [&](uint32_t off) { return reinterpret_cast<float*>(smem + off); };
    float* vm = f32(a.vm);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + a.misc);
    volatile int* s_ok = reinterpret_cast<volatile int*>(smem + a.misc + 8);

    // ---- weights; initial states; bias; first input: one trip to memory.  A staged vector holds BT values per
    // column and ends in zeros.
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
        mbar_expect_tx(bar, me.bytes);
        const uint8_t* src = a.images + (size_t)me.off16 * 16;
        for (uint32_t off = 0; off < me.bytes; off += 16384u) bulk_g2s(smem + off, src + off, min(16384u, me.bytes - off), bar);
        *s_ok = 1;
    }
    const uint32_t base = a.epoch[blockIdx.x] + 1u;        // the step number of step 0
    uint32_t above0 = 0;                                   // the progress of the layer above when this call began
    if (layer + 1 < a.L) above0 = ld_relaxed(a.progress + layer + 1);
    auto stage = [&](float* dst, const float* src, int n) {      // [B][n] in global memory
#pragma unroll 1
        for (int b = 0; b < BT; ++b)
#pragma unroll 2
            for (int i = tid; i < n; i += kR1Threads) dst[i * BT + b] = src && b < B ? __ldg(src + (size_t)b * n + i) : 0.f;
    };
    stage(f32(a.vr[1]), a.h0 ? a.h0 + (size_t)layer * B * S : nullptr, S);
    if (layer == 0) stage(f32(a.vu[0]), a.x, I);
    if (tid < 2 * BT) {
        const int b = tid & (BT - 1), k = tid / BT;
        f32(a.vr[0])[k * (int)(a.vr[1] - a.vr[0]) / 4 + S * BT + b] = 0.f;
        f32(a.vu[0])[k * (int)(a.vu[1] - a.vu[0]) / 4 + I * BT + b] = 0.f;
        if (OPS == 2) vm[H * BT + b] = 0.f;
    }
    if (layer == 0 && BT > 1)                                    // batch columns past B stay zero
#pragma unroll 1
        for (int i = tid; i < I * BT; i += kR1Threads) if (i % BT >= B) f32(a.vu[1])[i] = 0.f;
    // this lane's place: unit, row of the unit, batch column (the last lanes of a row share the columns when there are fewer)
    struct Lane { int unit, first_lane, row, sub, b; bool on, owner; float bias; } ln[OPS];
    const float* bl = a.bias[layer];
#pragma unroll
    for (int op = 0; op < OPS; ++op) {
        const int rows = op ? 1 : R0, lr_log = (op ? 5 : R0 == 4 ? 3 : 4) - me.lu[op], LR = 1 << lr_log;
        const int ui = lane / (rows * LR), u = (warp << me.lu[op]) + ui;
        Lane& l = ln[op];
        l.on = u < (int)me.units[op];
        l.unit = (int)me.unit0[op] + (l.on ? u : 0);
        l.first_lane = ui * rows * LR;
        l.sub = lane & (LR - 1);
        l.row = (lane >> lr_log) & (rows - 1);
        l.b = l.sub >> (lr_log - kBtLog);
        l.owner = l.on && l.row == 0 && (l.sub & ((LR >> kBtLog) - 1)) == 0;
        l.bias = 0.f;
        if (bl && l.on) {
            if (op == 0) l.bias = __ldg(bl + (size_t)l.row * H + l.unit);
            else if (CELL == kR1GruRb) l.bias = __ldg(bl + (size_t)2 * H + l.unit);
        }
    }
    float c = 0.f;                                         // cell state (reset-before GRU: the update gate) of the lane's unit and batch column
    if (kHasC && ln[0].on && a.c0 && ln[0].b < B) c = __ldg(a.c0 + ((size_t)layer * B + ln[0].b) * H + ln[0].unit);
    __syncthreads();
    bool ok = mbar_wait_bounded(bar, 0);
    if (!ok) *(volatile uint32_t*)a.status = (uint32_t)kDevCopyTimeout;
    RuWarp wd[OPS];
#pragma unroll
    for (int op = 0; op < OPS; ++op) wd[op] = reinterpret_cast<const RuWarp*>(smem)[op * kR1Warps + warp];

    // ---- the exchange: (value, step) pairs by element, kR1Ring steps of a vector
    const int n_state = S * BT, n_mid = H * BT;
    uint2* ex_state = a.ex[0][layer];
    uint2* ex_mid = a.ex[1][layer];
    const uint2* ex_below = layer > 0 ? a.ex[0][below] : nullptr;
    const int p_state = (n_state + 1) & ~1, p_mid = (n_mid + 1) & ~1;      // pitch of a step
    // Takes a vector: every thread asks for its pairs and asks again until they are of step `want`.
    auto take = [&](const uint2* src, int n, uint32_t want, float* dst) {
        want += a.never;
#pragma unroll 1
        for (int i0 = 2 * tid; i0 < n; i0 += 2 * kW * kR1Threads) {
            uint4 w[kW];
#pragma unroll
            for (int q = 0; q < kW; ++q) { const int i = i0 + 2 * q * kR1Threads; if (i < n) w[q] = ld_two(src + i); }
#pragma unroll
            for (int q = 0; q < kW; ++q) {
                const int i = i0 + 2 * q * kR1Threads;
                if (i < n) {
                    const bool two = i + 1 < n;
                    uint4 x = w[q];
                    if (x.y != want || (two && x.w != want)) {
                        x = wait_two(src + i, want, two, s_ok, a.status, a.limit_ns);
                        ok = ok && x.y == want && (!two || x.w == want);
                    }
                    // (the place behind the last element holds the vector's zero)
                    if (two) *reinterpret_cast<float2*>(dst + i) = make_float2(__uint_as_float(x.x), __uint_as_float(x.z));
                    else dst[i] = __uint_as_float(x.x);
                }
            }
        }
    };
    if (layer > 0) take(ex_below, n_state, base, f32(a.vu[0]));
    if (!__syncthreads_and(ok)) {
        if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
        return;
    }
#ifdef CSB_PHASE_CLOCKS
    long long lap[8] = {0, 0, 0, 0, 0, 0, 0, 0}, lap_at = clock64();
#endif
    // a product's lists of one part, and the sum over the lanes of a row: every lane gets the total of its row and batch column
    auto add_part = [&](int op, int part, const float* v, float (&acc)[BT]) {
        UnitWalk<T, BT>::run(smem + wd[op].off + (part ? (uint32_t)wd[op].n[0] * 512u : 0u) + lane * 16, wd[op].n[part], v, acc);
    };
    auto total = [&](float (&acc)[BT], int lr_log) {
        int off = 1 << (lr_log - 1);
#pragma unroll
        for (int h = BT / 2; h >= 1; h >>= 1, off >>= 1) {     // halve the batch columns a lane holds
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float give = up ? acc[i] : acc[i + h], keep = up ? acc[i + h] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
        }
#pragma unroll 1
        for (; off >= 1; off >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
        return acc[0];
    };
    const int lr0 = (R0 == 4 ? 3 : 4) - me.lu[0], lr1 = 5 - me.lu[1];
    size_t y_at = 0;                                       // where step t of the output starts
#pragma unroll 1
    for (int t = 0; t < T_; ++t, y_at += (size_t)B * S) {
        const bool more = t + 1 < T_;
        const float* vu = f32(a.vu[t & 1]);
        float* vu_next = f32(a.vu[(t + 1) & 1]);
        float* vr = f32(a.vr[(t + 1) & 1]);                // h_{t-1}
        const int ring = t & (kR1Ring - 1);
        if (layer == 0 && more) {
            const float* xs = a.x + (size_t)(t + 1) * B * I;
            // (a frame takes longer from memory than a step does: eight steps ahead into L2)
            if (t + 8 < T_ && tid * 32 < B * I) asm volatile("prefetch.global.L2 [%0];" ::"l"(xs + (size_t)7 * B * I + tid * 32));
#pragma unroll 1
            for (int b = 0; b < B; ++b)
#pragma unroll 1
                for (int i = tid; i < I; i += kR1Threads) cp_async4(vu_next + i * BT + b, xs + (size_t)b * I + i);
        }
        // ---- the input part, while h_{t-1} is on its way
        float acc[BT];
#pragma unroll
        for (int b = 0; b < BT; ++b) acc[b] = 0.f;
        add_part(0, 0, vu, acc);
        R1_LAP(0);                                         // product of the input part
        // the state of the step before and the next step's input, so that one barrier covers both
        if (a.L > 1) __nanosleep(kStatePause);
        if (t > 0) take(ex_state + (size_t)((t - 1) & (kR1Ring - 1)) * p_state, n_state, base + (uint32_t)(t - 1), vr);
        if (layer > 0 && more) take(ex_below + (size_t)((t + 1) & (kR1Ring - 1)) * p_state, n_state, base + (uint32_t)(t + 1), vu_next);
        if (layer == 0) cp_async_wait();
        // before the slots of steps t .. t + 7 are overwritten, the layer above must have read what they hold,
        // steps up to t - 25 (the count: see csb_rnn1_kernel.cuh)
        if (layer + 1 < a.L && t >= kR1Ring && (t & (kR1Block - 1)) == 0 && tid == kR1Threads - 1)
            ok = ok && wait_progress(a.progress + layer + 1, above0, (uint32_t)a.layer_ctas[layer + 1] * (uint32_t)((t - kR1Ring + kR1Block) / kR1Block), s_ok, a.status, a.limit_ns);
        R1_LAP(1);                                         // the state of the step before, the next input
        if (!__syncthreads_and(ok)) break;
        R1_LAP(2);
        if (layer > 0 && tid == 0 && (t & (kR1Block - 1)) == kR1Block - 1) atomicAdd(a.progress + layer, 1u);   // u up to step t has been read
        add_part(0, 1, vr, acc);
        const float z = total(acc, lr0) + ln[0].bias;
        R1_LAP(3);                                         // recurrent part, sums
        auto gate = [&](float v, int k) { return __shfl_sync(0xffffffffu, v, ln[0].first_lane + (k << lr0) + ln[0].sub); };
        float h;
        {
            const float hp = CELL == kR1Gru || CELL == kR1Ligru || CELL == kR1GruRb ? vr[ln[0].unit * BT + ln[0].b] : 0.f;
            if (kHasC) {
                const float y = activation(z, ln[0].row == 2);
                const float zi = gate(y, 0), zf = gate(y, 1), zc = gate(y, 2), zo = gate(y, 3);
                c = zf * c + zi * zc;
                h = zo * activation(c, true);
            } else if (CELL == kR1Gru) {
                const float y = activation(z, false);
                const float r = gate(y, 0), zz = gate(y, 1), ni = gate(z, 2), nh = gate(z, 3);
                h = (1.f - zz) * activation(ni + r * nh, true) + zz * hp;
            } else if (CELL == kR1Ligru) {
                const float zz = gate(activation(z, false), 0), cand = fmaxf(gate(z, 1), 0.f);
                h = zz * hp + (1.f - zz) * cand;
            } else {
                const float y = activation(z, false);
                h = gate(y, 0) * hp;                       // r * h_{t-1}
                c = gate(y, 1);
            }
        }
        if (OPS == 1) {
            if (ln[0].owner) {
                if (more || layer + 1 < a.L) st_one(ex_state + (size_t)ring * p_state + ln[0].unit * BT + ln[0].b, h, base + (uint32_t)t);
                if (ln[0].b < B) {
                    const size_t at = (size_t)ln[0].b * S + ln[0].unit;
                    if (layer == a.L - 1 && a.y) a.y[y_at + at] = h;
                    if (!more && a.hT) a.hT[(size_t)layer * B * S + at] = h;
                }
            }
        } else {
            if (ln[0].owner) st_one(ex_mid + (size_t)ring * p_mid + ln[0].unit * BT + ln[0].b, h, base + (uint32_t)t);
        }
        if (kHasC && !more && a.cT && ln[0].owner && ln[0].b < B) a.cT[((size_t)layer * B + ln[0].b) * H + ln[0].unit] = c;
        R1_LAP(5);                                         // gates
        if (OPS == 2) {
            // ---- second product of the step: what the first one gave, from every CTA of the layer
#pragma unroll
            for (int b = 0; b < BT; ++b) acc[b] = 0.f;
            if (CELL == kR1GruRb) add_part(OPS - 1, 0, vu, acc);
            __nanosleep(kMidPause);
            take(ex_mid + (size_t)ring * p_mid, n_mid, base + (uint32_t)t, vm);
            if (!__syncthreads_and(ok)) break;
            R1_LAP(6);                                     // exchange inside the step
            add_part(OPS - 1, 1, vm, acc);
            float s = total(acc, lr1) + ln[OPS - 1].bias;
            const Lane& l = ln[OPS - 1];
            if (CELL == kR1GruRb) {
                // (a unit has the same lanes in both products, its batch columns another spacing)
                const float zz = __shfl_sync(0xffffffffu, c, l.first_lane + (l.b << (lr0 - kBtLog)));
                s = (1.f - zz) * activation(s, true) + zz * vr[l.unit * BT + l.b];
            }
            if (l.owner) {
                if (more || layer + 1 < a.L) st_one(ex_state + (size_t)ring * p_state + l.unit * BT + l.b, s, base + (uint32_t)t);
                if (l.b < B) {
                    const size_t at = (size_t)l.b * S + l.unit;
                    if (layer == a.L - 1 && a.y) a.y[y_at + at] = s;
                    if (!more && a.hT) a.hT[(size_t)layer * B * S + at] = s;
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

template <typename T, int BT>
static const void* pick_unit_kernel(int cell) {
    switch (cell) {
        case kR1Lstm: return (const void*)csb_rnn_unit_kernel<T, kR1Lstm, BT>;
        case kR1Gru: return (const void*)csb_rnn_unit_kernel<T, kR1Gru, BT>;
        case kR1Lstmp: return (const void*)csb_rnn_unit_kernel<T, kR1Lstmp, BT>;
        case kR1Ligru: return (const void*)csb_rnn_unit_kernel<T, kR1Ligru, BT>;
        default: return (const void*)csb_rnn_unit_kernel<T, kR1GruRb, BT>;
    }
}

}  // namespace csb
