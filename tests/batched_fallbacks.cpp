// The host side of the batched recurrent calls (csb_umma_rnn.cu, csb_rnn_step.cu) on the CUDA runtime of fake_runtime.hpp: where
// the time loop cannot run, the call has to be left to the step-by-step form, and that form has to refuse a handle
// whose product gave up.  Exit code 0: every rule below held.
#include "../paper_2005_05758_b200/csrc/csb_umma_rnn.hpp"
#include "fake_runtime.hpp"

using namespace csb;

static int g_clusters = 148;                               // CTAs that the device holds at a time
namespace csb {
void set_error(const char*, ...) {}
void clear_error() {}
int umma_clusters(const csb_matrix*, int (&n)[kUmmaMaxS + 1]) {
    for (int s = 0; s <= kUmmaMaxS; ++s) n[s] = s ? g_clusters / s : 0;
    return CSB_OK;
}
const void* pick_umma(int, int, int) { return nullptr; }
bool umma_stages(int, int, int, int max_round, size_t room, UmmaStages* out) { *out = UmmaStages{2, max_round, room}; return true; }
static int g_products = 0, g_other_products = 0;
int launch_umma_fp32(const csb_matrix*, const UmmaPlan*, uint8_t*, const float*, int64_t, int, float*, int64_t, cudaStream_t) { ++g_products; return CSB_OK; }
bool spmm_mma_applicable(const csb_matrix*, int) { return true; }
int prepare_spmm_stack(int, const csb_matrix* const*, int, SpmmStack*) { return CSB_OK; }
int launch_spmm_stack(const SpmmStack&, int, int, const csb_matrix* const*, uint8_t* const*, float* const*, int, int64_t, void*) { return CSB_ERR_LAUNCH; }
int launch_spmm_stack_fp32(const SpmmStack&, int, const csb_matrix*, uint8_t*, const float*, int64_t, int, float*, int64_t, void*) { ++g_other_products; return CSB_OK; }
void note_recurrent_path(RecurrentPath) {}
void note_tensor_kernel(TensorKernel) {}
void barrier_test_hook(unsigned int* extra, unsigned long long* ns) { *extra = 0; *ns = 1; }
}

static const int I = 70, H = 96, L = 2, T = 3, B = 20, block = 32;
static csb_matrix* layer(int cols, uint64_t uid) {
    std::vector<float> W((size_t)4 * H * cols, 1.f);
    const size_t blocks = (size_t)(4 * H / block) * ((cols + block - 1) / block);
    std::vector<uint8_t> rk(blocks * block, 1), ck(rk.size(), 1);
    csb_matrix* A = new csb_matrix();
    A->device = 0; A->smem_optin = 232448; A->uid = uid;
    if (encode_host(W.data(), 4 * H, cols, cols, block, block, rk.data(), ck.data(), CSB_F16, A) != CSB_OK) std::exit(3);
    return A;
}

int main() {
    csb_matrix* W[L] = {layer(I + H, 1), layer(2 * H, 2)};
    const int in_size[L] = {I, H};
    std::vector<float> x((size_t)T * B * I), y((size_t)T * B * H), s((size_t)L * B * H);
    auto call = [&](unsigned flags) {
        return rnn_forward_umma(4, L, W, nullptr, x.data(), T, B, H, in_size, s.data(), s.data(), y.data(), nullptr, nullptr, flags, nullptr);
    };
    auto forget = [&](const char* what, long n) {
        for (csb_matrix* A : W) drop_umma_rnn_plans(A);
        const int left = (int)g_live.size();
        if (left) printf("%s, call %ld: %d arrays left\n", what, n, left);
        g_live.clear();
        return left != 0;
    };
    int bad = 0;
    for (int onwards = 0; onwards < 2; ++onwards)
        for (long n = 0;; ++n) {
            g_calls = 0; g_fails = n; g_onwards = onwards;
            const int rc = call(0);
            const bool failed = g_calls > n;
            // (the last call that can fail is the one that waits for the result)
            if (failed ? rc != 1 && rc != CSB_ERR_ALLOC : rc != CSB_OK) { printf("call %ld: status %d\n", n, rc); ++bad; }
            if (rc == CSB_ERR_ALLOC && g_launches < 2) { printf("call %ld: refused before anything ran\n", n); ++bad; }
            g_fails = -1;
            const int again = call(0);
            if (again != CSB_OK && again != 1) { printf("call %ld: then status %d\n", n, again); ++bad; }
            bad += forget("out of memory", n);
            g_launches = 0;
            if (!failed) break;
        }
    g_cooperative = cudaErrorCooperativeLaunchTooLarge;
    const int large = call(0);
    if (large != 1) { printf("a grid that does not fit: status %d\n", large); ++bad; }
    g_cooperative = cudaSuccess;
    if (call(0) != CSB_OK) { puts("and then"); ++bad; }
    bad += forget("grid", 0);
    // a stack that one grid does not hold: nothing is laid out for a loop that never runs
    g_clusters = 2; g_bytes = 0;
    if (call(0) != 1 || g_bytes) { printf("a stack past the grid: %zu bytes\n", g_bytes); ++bad; }
    std::shared_ptr<UmmaStack> stack;                      // but for fp32 buffers, which use the layouts step by step
    if (umma_stack(4, L, W, in_size, H, false, &stack) != CSB_OK || !stack || !stack->plan[L - 1].d_stream) { puts("no layouts for the fp32 buffers"); ++bad; }
    if (call(0) != 1) { puts("a stack past the grid, laid out"); ++bad; }
    stack.reset();
    bad += forget("past the grid", 0);
    // more sequences than the loop takes: step by step, and no step with a handle whose product has given up
    g_clusters = 148;
    const int many = 40;
    std::vector<float> xs((size_t)T * many * I), ys((size_t)T * many * H), ss((size_t)L * many * H);
    auto steps = [&]() {
        g_products = g_other_products = 0;
        return rnn_forward_stepwise(4, L, W, nullptr, xs.data(), T, many, H, in_size, ss.data(), ss.data(), ys.data(), nullptr, nullptr, CSB_FLAG_ASYNC, nullptr);
    };
    if (steps() != CSB_OK || g_products != T * L) { printf("steps: %d products\n", g_products); ++bad; }
    uint32_t word = 1;
    W[0]->product.h_status = &word;
    if (steps() != CSB_ERR_TIMEOUT || g_products) { printf("steps of a handle that gave up: %d products\n", g_products); ++bad; }
    W[0]->product.h_status = nullptr;
    // the environment is read at every call: a plan of one form does not serve the other
    setenv("CSB_NO_UMMA", "1", 1);
    if (steps() != CSB_OK || g_products || g_other_products != T * L) { printf("steps by mma.sync: %d products, %d others\n", g_products, g_other_products); ++bad; }
    unsetenv("CSB_NO_UMMA");
    if (steps() != CSB_OK || g_products != T * L || g_other_products) { printf("steps again: %d products, %d others\n", g_products, g_other_products); ++bad; }
    for (csb_matrix* A : W) drop_step_plans(A);
    bad += forget("steps", 0);
    puts(bad ? "failed" : "ok");
    return bad != 0;
}
