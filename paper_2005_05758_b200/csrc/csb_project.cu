// Projection of a dense weight onto the CSB pattern: the RowPrune / ColumnPrune step of the
// paper's Algorithm 1 (Section 3.2), which turns any dense matrix and a target pruning rate into
// the per-block row and column keep masks that csb_encode takes.
//
// RowPrune works on every block-column on its own: the squared l2-norm of each row segment (the
// part of a matrix row inside the block-column) is taken and the weakest fraction p of the
// segments is pruned; ColumnPrune then does the same with the column segments of every block-row
// of the result.  p = 1 - sqrt(1 - PR), so about PR of the weights are gone after both.
//
// Four launches on one stream, each ordered behind the one in front by programmatic dependent launch:
// norms of the row segments (one pass over the weight, fp64 sums), selection per block-column, norms
// of the column segments (the surviving half of the rows once more), selection per block-row.
//
// Bound by memory, 0.40 GB for 8192 x 8192 at 0.75.  Measured there: 88.5 us a call (166.4 with a thread
// per row segment, 16 bytes of every 256 per load, and radix selections); the row pass reads at 5.4
// TB/s, the column pass at 4.2 TB/s (profiler, cold caches).  Chunks of block-columns, so that the column
// pass finds its rows in L2, were slower: eleven short launches, 207 us.
#include <algorithm>

#include "csb_internal.hpp"
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

constexpr int kNormWarps = 8, kSelThreads = 1024;
constexpr int64_t kMaxSelect = 20480;          // segments per selection (rows or columns of the weight)
constexpr int kSelKeys = 8;                    // keys a thread keeps in registers: 8192 segments, more are read again
constexpr int kSelBuckets = 2048, kSelCand = 1024;

struct ProjectArgs {
    const float* W;
    long long ld;
    int R, C, BR, BC, nbr, nbc;
    double* rn;                                // [nbc, R] norms of the row segments
    double* cn;                                // [nbr, C] norms of the column segments
    uint8_t* row_keep;
    uint8_t* col_keep;
    unsigned int k_rows, k_cols;               // segments pruned per block-column / block-row
};

// E consecutive columns from p, as far as they exist (`left` columns from p on, at least one): the
// loads are unconditional, so that many go out together, and what lies past the edge reads the last
// existing piece again and is counted as zero.
template <int E> struct Piece { float v[E]; };
template <int E>
__device__ __forceinline__ Piece<E> load_piece(const float* p) {
    Piece<E> r;
    if (E == 4) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(p));
        r.v[0] = t.x; r.v[E > 1 ? 1 : 0] = t.y; r.v[E > 2 ? 2 : 0] = t.z; r.v[E > 3 ? 3 : 0] = t.w;
    } else {
        r.v[0] = __ldg(p);
    }
    return r;
}

// Norms of the row segments.  LW lanes (a power of two) share a segment, a lane takes E columns of it
// at a time (4 with 16-byte loads when rows and blocks are aligned, else 1), so every load instruction
// reads consecutive floats.  A warp works on 16 * 32 / LW rows of one block-column with 16 loads in
// flight per lane (E = 4: 8 KB per warp), neighbouring warps on neighbouring block-columns.  The
// lanes' partial sums are folded for several rows at once: in each round a lane keeps half of its
// rows and hands over the other half, so FV rows over LW lanes cost FV - 1 exchanges (and
// log2(LW / FV) more) instead of FV log2 LW.
template <int E, int LW>
__global__ void __launch_bounds__(kNormWarps * 32, 2) csb_row_segment_norms_kernel(const ProjectArgs a) {
    constexpr int V = 16, FV = LW < V ? LW : V;
    pdl_launch_dependents();
    pdl_wait();
    const int lane = threadIdx.x & 31, grp = lane / LW, gl = lane % LW;
    const unsigned int u = blockIdx.x * kNormWarps + (threadIdx.x >> 5);
    const int rb = (int)(u / (unsigned)a.nbc), bj = (int)(u - (unsigned)rb * (unsigned)a.nbc);
    const int r0 = rb * (V * (32 / LW)) + grp * V;
    if (rb * (V * (32 / LW)) >= a.R) return;
    const int c0 = bj * a.BC, nc = min(a.BC, a.C - c0);
    double s[V];
#pragma unroll
    for (int v = 0; v < V; ++v) s[v] = 0.0;
    size_t row[V];
#pragma unroll
    for (int v = 0; v < V; ++v) row[v] = (size_t)min(r0 + v, a.R - 1) * a.ld;
    auto sweep = [&](int c, bool all) {
        const bool in = all || c + gl * E < nc;            // E divides nc
        const float* p = a.W + c0 + (all ? c + gl * E : min(c + gl * E, nc - E));
        Piece<E> x[V];
#pragma unroll
        for (int v = 0; v < V; ++v) x[v] = load_piece<E>(p + row[v]);
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int e = 0; e < E; ++e) { const double d = in ? x[v].v[e] : 0.f; s[v] = fma(d, d, s[v]); }
    };
    int c = 0;
    for (; c + LW * E <= nc; c += LW * E) sweep(c, true);
    if (c < nc) sweep(c, false);
#pragma unroll
    for (int f = 0; f < V; f += FV) {
#pragma unroll
        for (int h = FV / 2, off = LW / 2; h >= 1; h >>= 1, off >>= 1) {
            const bool up = (gl & off) != 0;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const double give = up ? s[f + i] : s[f + i + h], keep = up ? s[f + i + h] : s[f + i];
                s[f + i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
        }
#pragma unroll
        for (int off = LW / FV / 2; off >= 1; off >>= 1) s[f] += __shfl_xor_sync(0xffffffffu, s[f], off);
        // the lane's bits LW/2, LW/4, ... say which row's sum it holds, highest bit first
        const int r = r0 + f + gl / (LW / FV);
        if (gl % (LW / FV) == 0 && r < a.R) a.rn[(size_t)bj * a.R + r] = s[f];
    }
}

// Norms of the column segments after RowPrune.  A warp works on one block: LW lanes cover a row of it
// (E columns each; wider blocks in several sweeps), the 32 / LW lane groups take the surviving rows in
// turn, eight rows' loads go out together, and the groups' sums are
// added at the end.  Blocks are taken last to first: what the first pass read last is still in L2.
template <int E, int LW>
__global__ void __launch_bounds__(kNormWarps * 32, 3) csb_col_segment_norms_kernel(const ProjectArgs a) {
    constexpr int G = 32 / LW;
    pdl_launch_dependents();
    pdl_wait();
    const int lane = threadIdx.x & 31, grp = lane / LW, gl = lane % LW;
    const unsigned int n = (unsigned)a.nbr * (unsigned)a.nbc, w = blockIdx.x * kNormWarps + (threadIdx.x >> 5);
    if (w >= n) return;
    const unsigned int u = n - 1u - w;
    const int bi = (int)(u / (unsigned)a.nbc), bj = (int)(u - (unsigned)bi * (unsigned)a.nbc);
    const int r0 = bi * a.BR, nr = min(a.BR, a.R - r0), c0 = bj * a.BC, nc = min(a.BC, a.C - c0);
    const uint8_t* flags = a.row_keep + (size_t)u * a.BR;
    // the surviving rows as a list, so that the lane groups share them evenly and no load is wasted
    __shared__ uint8_t s_rows[kNormWarps][256];
    uint8_t* list = s_rows[threadIdx.x >> 5];
    int kept = 0;
    for (int rb = 0; rb < nr; rb += 32) {
        const bool f = rb + lane < nr && __ldcg(flags + rb + lane) != 0;
        const unsigned int m = __ballot_sync(0xffffffffu, f);
        if (f) list[kept + __popc(m & ((1u << lane) - 1u))] = (uint8_t)(rb + lane);
        kept += __popc(m);
    }
    __syncwarp();
    for (int c = 0; c < nc; c += LW * E) {
        const bool in = c + gl * E < nc;
        const float* p = a.W + (size_t)r0 * a.ld + c0 + min(c + gl * E, nc - E);
        double s[E];
#pragma unroll
        for (int e = 0; e < E; ++e) s[e] = 0.0;
        auto batch = [&](int i0, bool all) {
            Piece<E> x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = load_piece<E>(p + (size_t)list[all ? i0 + j * G : min(i0 + j * G, kept - 1)] * a.ld);
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int e = 0; e < E; ++e) { const double d = all || i0 + j * G < kept ? x[j].v[e] : 0.f; s[e] = fma(d, d, s[e]); }
        };
        int i = 0;
        for (; i + 8 * G <= kept; i += 8 * G) batch(i + grp, true);
        if (i < kept) batch(i + grp, false);
#pragma unroll
        for (int off = LW; off < 32; off <<= 1)
#pragma unroll
            for (int e = 0; e < E; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], off);
        if (grp == 0 && in) {
            double* out = a.cn + (size_t)bi * a.C + c0 + c + gl * E;
#pragma unroll
            for (int e = 0; e < E; ++e) out[e] = s[e];
        }
    }
}

// Shared memory of a selection.
struct SelectSmem {
    unsigned int hist[kSelBuckets];
    unsigned long long cand[kSelCand];
    unsigned int cand_idx[kSelCand];
    unsigned int red[2 * (kSelThreads / 32)];
    unsigned long long sel[2];
    unsigned int n_cand;
};

// k-th smallest (1-based) of the keys that pass `pred`, by 8-bit radix passes from the top; returns
// the key and, through rank_in_equals, how many of the keys equal to it are among the k smallest.
// The way for groups with many ties or non-finite norms.  All threads of the CTA call it.
template <typename Key, int BYTES, typename Get, typename Pred>
__device__ Key radix_select(int n, unsigned int k, Get get, Pred pred, unsigned int* hist, unsigned long long* sel,
                            unsigned int* rank_in_equals) {
    Key prefix = 0, mask = 0;
    for (int shift = 8 * (BYTES - 1); shift >= 0; shift -= 8) {
        for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0u;
        __syncthreads();
        for (int i0 = 0; i0 < n; i0 += blockDim.x) {
            const int i = i0 + threadIdx.x;
            unsigned int bucket = 0xffffffffu;
            if (i < n && pred(i)) {
                const Key key = get(i);
                if ((key & mask) == prefix) bucket = (unsigned int)((key >> shift) & (Key)255);
            }
            // nearly all keys may share a bucket: lanes of a warp that hit the same one add once, together
            const unsigned int peers = __match_any_sync(0xffffffffu, bucket);
            if (bucket != 0xffffffffu && (threadIdx.x & 31) == (unsigned)(__ffs(peers) - 1)) atomicAdd(&hist[bucket], (unsigned int)__popc(peers));
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // warp 0 finds the bucket where the running count reaches k: eight buckets per lane
            const unsigned int lane = threadIdx.x;
            unsigned int mine = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) mine += hist[lane * 8 + j];
            unsigned int incl = mine;
            for (int off = 1; off < 32; off <<= 1) { const unsigned int o = __shfl_up_sync(0xffffffffu, incl, off); if (lane >= (unsigned)off) incl += o; }
            const unsigned int before = incl - mine;
            const unsigned int hit = __ballot_sync(0xffffffffu, incl >= k);
            if (lane == (unsigned)(__ffs(hit) - 1)) {
                unsigned int cum = before, b = lane * 8;
                for (int j = 0; j < 7; ++j, ++b) { if (cum + hist[b] >= k) break; cum += hist[b]; }
                sel[0] = b; sel[1] = k - cum;
            }
        }
        __syncthreads();
        prefix |= (Key)sel[0] << shift;
        mask |= (Key)255 << shift;
        k = (unsigned int)sel[1];
        __syncthreads();
    }
    *rank_in_equals = k;
    return prefix;
}

// One CTA per group (a block-column's row segments, or a block-row's column segments): prune the k
// weakest of its n segments and write the keep flags where csb_encode expects them (flags of in-block
// lines beyond the matrix edge are 0).  Among equal norms the highest index goes first.
//   ROWS: group g is block-column g, segment s is matrix row s   -> row_keep[((s / B) * nbc + g) * B + s % B]
//   else: group g is block-row g, segment s is matrix column s   -> col_keep[(g * nbc + s / B) * B + s % B]
//
// Norms of a group lie within a factor of a few, so they are counted in 2048 equal steps between (just
// below) the smallest and (just above) the largest: (v - lowest) times a constant, rounded, never
// decreases in v.  Only the keys in the step that holds the k-th are ranked against each other; the
// others' steps decide for them.  8192 segments, 128 groups: 12 us against 28 us for eight
// radix passes (both under the profiler, cold caches).
template <bool ROWS>
__global__ void __launch_bounds__(kSelThreads, 1) csb_select_prune_kernel(const ProjectArgs a) {
    __shared__ SelectSmem S;
    constexpr int kWarps = kSelThreads / 32;
    static_assert(kWarps == 32, "one lane per warp's result");
    const int g = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n = ROWS ? a.R : a.C, B = ROWS ? a.BR : a.BC, nblk = ROWS ? a.nbr : a.nbc;
    const unsigned int k = ROWS ? a.k_rows : a.k_cols;
    const double* norms = (ROWS ? a.rn : a.cn) + (size_t)g * n;
    for (int i = t; i < kSelBuckets; i += kSelThreads) S.hist[i] = 0u;
    if (t == 0) S.n_cand = 0u;
    pdl_launch_dependents();
    pdl_wait();
    const bool cached = n <= kSelKeys * kSelThreads;
    // sums of squares are >= +0, so the bit patterns order like the values
    unsigned long long key[kSelKeys];
#pragma unroll
    for (int j = 0; j < kSelKeys; ++j) {
        const int i = t + j * kSelThreads;
        key[j] = cached && i < n ? (unsigned long long)__double_as_longlong(__ldcg(norms + i)) : 0ull;
    }
    auto get = [&](int i) { return (unsigned long long)__double_as_longlong(__ldcg(norms + i)); };
    auto each = [&](auto f) {
        if (cached) {
#pragma unroll
            for (int j = 0; j < kSelKeys; ++j) {
                const int i = t + j * kSelThreads;
                if (i < n) f(i, key[j]);
            }
        } else {
            for (int i = t; i < n; i += kSelThreads) f(i, get(i));
        }
    };
    // smallest and largest upper word
    unsigned int lo = 0xffffffffu, hi = 0u;
    each([&](int, unsigned long long x) { const unsigned int w = (unsigned int)(x >> 32); lo = min(lo, w); hi = max(hi, w); });
    lo = __reduce_min_sync(0xffffffffu, lo); hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { S.red[warp] = lo; S.red[kWarps + warp] = hi; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, S.red[lane]); hi = __reduce_max_sync(0xffffffffu, S.red[kWarps + lane]);
    const double lowest = __hiloint2double((int)lo, 0), range = __hiloint2double((int)hi + 1, 0) - lowest;
    const float scale = (float)kSelBuckets / (float)range;
    auto step_of = [&](unsigned long long x) { return min(kSelBuckets - 1, (int)((float)(__longlong_as_double((long long)x) - lowest) * scale)); };
    int b_cut = -1;                                        // steps below it go, steps above it stay
    unsigned long long v = 0ull;                           // inside it: keys below v, and those equal to v from idx_cut on
    unsigned int idx_cut = 0xffffffffu;
    bool by_step = range > 1e-30 && range < 1e30;          // false for (nearly) all equal, infinite, NaN
    if (k > 0 && by_step) {
        each([&](int, unsigned long long x) { atomicAdd(&S.hist[step_of(x)], 1u); });
        __syncthreads();
        // the step where the running count reaches k: two steps per thread
        constexpr int kPer = kSelBuckets / kSelThreads;
        unsigned int h[kPer], mine = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) { h[j] = S.hist[t * kPer + j]; mine += h[j]; }
        unsigned int incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) { const unsigned int o = __shfl_up_sync(0xffffffffu, incl, off); if (lane >= off) incl += o; }
        if (lane == 31) S.red[warp] = incl;
        __syncthreads();
        unsigned int cum = incl - mine + __reduce_add_sync(0xffffffffu, lane < warp ? S.red[lane] : 0u);
        if (cum < k && cum + mine >= k) {
            int b = 0;
            while (cum + h[b] < k) { cum += h[b]; ++b; }
            S.sel[0] = (unsigned long long)(t * kPer + b); S.sel[1] = k - cum;
        }
        __syncthreads();
        b_cut = (int)S.sel[0];
        const unsigned int need = (unsigned int)S.sel[1];
        by_step = S.hist[b_cut] <= (unsigned int)kSelCand;
        if (by_step) {
            each([&](int i, unsigned long long x) {
                if (step_of(x) == b_cut) { const unsigned int at = atomicAdd(&S.n_cand, 1u); S.cand[at] = x; S.cand_idx[at] = (unsigned int)i; }
            });
            __syncthreads();
            const int nc = (int)S.n_cand;
            for (int i = t; i < nc; i += kSelThreads) {
                const unsigned long long x = S.cand[i];
                const unsigned int idx = S.cand_idx[i];
                unsigned int before = 0;
                for (int j = 0; j < nc; ++j) before += S.cand[j] < x || (S.cand[j] == x && S.cand_idx[j] > idx);
                if (before == need - 1u) { S.sel[0] = x; S.red[0] = idx; }
            }
            __syncthreads();
            v = S.sel[0];
            idx_cut = S.red[0];
        }
    }
    if (k > 0 && !by_step) {
        __syncthreads();
        unsigned int need = 0, dummy = 0;
        v = radix_select<unsigned long long, 8>(n, k, get, [&](int) { return true; }, S.hist, S.sel, &need);
        // the `need` highest indices among the ties: the need-th smallest of the inverted indices
        idx_cut = 0xffffffffu - radix_select<unsigned int, 4>(n, need, [&](int i) { return 0xffffffffu - (unsigned int)i; },
                                                              [&](int i) { return get(i) == v; }, S.hist, S.sel, &dummy);
    }
    // block and place of this thread's segments, followed from one to the next without dividing
    uint8_t* keep = ROWS ? a.row_keep + (size_t)g * B : a.col_keep + (size_t)g * a.nbc * B;
    const size_t pitch = ROWS ? (size_t)a.nbc * B : (size_t)B;
    const int blk_step = kSelThreads / B, at_step = kSelThreads - blk_step * B;
    int blk = t / B, at = t - blk * B;
    auto put = [&](bool kept) {
        keep[blk * pitch + at] = kept ? 1 : 0;
        blk += blk_step; at += at_step;
        if (at >= B) { at -= B; ++blk; }
    };
    each([&](int i, unsigned long long x) {
        const int b = by_step ? step_of(x) : b_cut;
        put(k == 0 || b > b_cut || (b == b_cut && !(x < v || (x == v && (unsigned int)i >= idx_cut))));
    });
    while (blk < nblk) put(false);
}

static unsigned int pruned_count(double p, int64_t n) {
    const double v = p * (double)n + 0.5;
    return (unsigned int)std::min<double>((double)n, v < 0 ? 0.0 : std::floor(v));
}

// The norm kernels for a block width: the fewest lanes (a power of two) that cover a block with E columns each.
typedef void (*ProjectKernel)(const ProjectArgs);
struct NormKernels { ProjectKernel rows, cols; int lanes; };
template <int E, int LW>
static NormKernels norm_kernels() { return {csb_row_segment_norms_kernel<E, LW>, csb_col_segment_norms_kernel<E, LW>, LW}; }
static NormKernels pick_norm_kernels(bool vec, int BC) {
    if (vec) return BC <= 16 ? norm_kernels<4, 4>() : BC <= 32 ? norm_kernels<4, 8>() : BC <= 64 ? norm_kernels<4, 16>() : norm_kernels<4, 32>();
    return BC <= 8 ? norm_kernels<1, 8>() : BC <= 16 ? norm_kernels<1, 16>() : norm_kernels<1, 32>();
}

int project_device(const float* W, int64_t R, int64_t C, int64_t ld, int BR, int BC, double PR, uint8_t* row_keep,
                   uint8_t* col_keep, void* workspace, int64_t workspace_bytes, void* stream) {
    const int64_t nbr = (R + BR - 1) / BR, nbc = (C + BC - 1) / BC;
    const int64_t need = (nbc * R + nbr * C) * 8;
    if (workspace_bytes < need) { set_error("workspace of %lld bytes, %lld needed", (long long)workspace_bytes, (long long)need); return CSB_ERR_INVALID_ARG; }
    if (R > kMaxSelect || C > kMaxSelect) { set_error("rows and columns above %lld are not supported by the selection kernel", (long long)kMaxSelect); return CSB_ERR_UNSUPPORTED; }
    const double p = 1.0 - std::sqrt(1.0 - PR);
    ProjectArgs a{};
    a.W = W; a.ld = ld; a.R = (int)R; a.C = (int)C; a.BR = BR; a.BC = BC; a.nbr = (int)nbr; a.nbc = (int)nbc;
    a.rn = reinterpret_cast<double*>(workspace); a.cn = a.rn + nbc * R;
    a.row_keep = row_keep; a.col_keep = col_keep;
    a.k_rows = pruned_count(p, R); a.k_cols = pruned_count(p, C);
    // 16-byte loads need aligned rows, and blocks and edges that end on them
    const bool vec = (reinterpret_cast<uintptr_t>(W) & 15) == 0 && ld % 4 == 0 && BC % 4 == 0 && C % 4 == 0;
    const NormKernels K = pick_norm_kernels(vec, BC);
    const int64_t row_units = nbc * ((R + 512 / K.lanes - 1) / (512 / K.lanes)), col_units = nbc * nbr;
    struct Launch { ProjectKernel kernel; int64_t ctas; int threads; };
    const Launch steps[4] = {{K.rows, (row_units + kNormWarps - 1) / kNormWarps, kNormWarps * 32},
                             {csb_select_prune_kernel<true>, nbc, kSelThreads},
                             {K.cols, (col_units + kNormWarps - 1) / kNormWarps, kNormWarps * 32},
                             {csb_select_prune_kernel<false>, nbr, kSelThreads}};
    for (const Launch& l : steps) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)l.ctas); cfg.blockDim = dim3((unsigned)l.threads); cfg.stream = (cudaStream_t)stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        CSB_CUDA(cudaLaunchKernelEx(&cfg, l.kernel, a));
    }
    CSB_CUDA(cudaGetLastError());
    return CSB_OK;
}

}  // namespace csb

extern "C" {

int64_t csb_project_workspace_bytes(int64_t rows, int64_t cols, int block_r, int block_c) {
    if (rows <= 0 || cols <= 0 || block_r < 1 || block_c < 1) return 0;
    const int64_t nbr = (rows + block_r - 1) / block_r, nbc = (cols + block_c - 1) / block_c;
    return (nbc * rows + nbr * cols) * 8;
}

int csb_project(const float* dense, int64_t rows, int64_t cols, int64_t ld, int block_r, int block_c, double prune_fraction,
                uint8_t* row_keep, uint8_t* col_keep, void* workspace, int64_t workspace_bytes, void* stream) {
    csb::clear_error();
    if (!dense || !row_keep || !col_keep || !workspace) { csb::set_error("dense, row_keep, col_keep or workspace is NULL"); return CSB_ERR_INVALID_ARG; }
    if (rows <= 0 || cols <= 0 || ld < cols) { csb::set_error("rows=%lld cols=%lld ld=%lld", (long long)rows, (long long)cols, (long long)ld); return CSB_ERR_INVALID_ARG; }
    if (block_r < 1 || block_r > 256 || block_c < 1 || block_c > 256) { csb::set_error("block sizes must be 1..256, got %dx%d", block_r, block_c); return CSB_ERR_INVALID_ARG; }
    if (!(prune_fraction >= 0.0 && prune_fraction <= 1.0)) { csb::set_error("prune_fraction %g is outside [0, 1]", prune_fraction); return CSB_ERR_INVALID_ARG; }
    return csb::project_device(dense, rows, cols, ld, block_r, block_c, prune_fraction, row_keep, col_keep, workspace, workspace_bytes, stream);
}

}  // extern "C"
