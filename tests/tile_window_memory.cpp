// The device side of a plan of the batched product (csb_umma_upload.cpp) on the CUDA runtime of fake_runtime.hpp, whose
// n-th call that can fail does so, once or from then on, for every n.  Exit code 0: every rule below held.
#include "../paper_2005_05758_b200/csrc/csb_umma_rnn.hpp"
#include "fake_runtime.hpp"

using namespace csb;

namespace csb {
void set_error(const char*, ...) {}
void clear_error() {}
int umma_clusters(const csb_matrix*, int (&n)[kUmmaMaxS + 1]) {
    for (int s = 0; s <= kUmmaMaxS; ++s) n[s] = s ? 148 / s : 0;
    return CSB_OK;
}
const void* pick_umma(int, int, int) { return nullptr; }
bool umma_stages(int, int, int, int max_round, size_t room, UmmaStages* out) { *out = UmmaStages{2, max_round, room}; return true; }
}

static bool whole(const UmmaPlan& P) { return P.d_stream && P.d_ctas && P.d_quads && P.d_rounds && P.d_xp; }

int main() {
    const int R = 300, C = 200, b = 32;
    std::vector<float> W((size_t)R * C, 1.f);
    std::vector<uint8_t> rk(10 * 7 * b, 1), ck(rk.size(), 1);
    csb_matrix A;
    A.smem_optin = 232448;
    if (encode_host(W.data(), R, C, C, b, b, rk.data(), ck.data(), CSB_F16, &A) != CSB_OK) return 3;
    int bad = 0;
    for (int onwards = 0; onwards < 2; ++onwards)
        for (const cudaError_t error : {cudaErrorMemoryAllocation, cudaErrorStreamCaptureUnsupported})
            for (long n = 0;; ++n) {
                UmmaPlan P;
                g_calls = 0; g_fails = n; g_onwards = onwards; g_error = error;
                const int rc = make_umma_plan(&A, &P);
                const bool failed = g_calls > n;
                // a plan that counts as built has all of its arrays, one that does not has none
                if (P.built ? !whole(P) : !g_live.empty()) { printf("call %ld: built %d, %zu arrays\n", n, P.built, g_live.size()); ++bad; }
                // out of memory: the other form takes the matrix, at once and from then on; any other failure is reported, once
                const int want = !failed ? (int)CSB_OK : error == cudaErrorMemoryAllocation ? 1 : (int)CSB_ERR_CUDA;
                if (rc != want) { printf("call %ld: status %d, not %d\n", n, rc, want); ++bad; }
                g_fails = -1;
                const int again = make_umma_plan(&A, &P), then = failed && error == cudaErrorMemoryAllocation ? 1 : (int)CSB_OK;
                if (again != then || P.built != (then == CSB_OK) || (P.built && !whole(P))) { printf("call %ld: then status %d, built %d\n", n, again, P.built); ++bad; }
                drop_umma_plan(P);
                if (!g_live.empty()) { printf("call %ld: %zu arrays left\n", n, g_live.size()); ++bad; g_live.clear(); }
                if (!failed) break;
            }
    puts(bad ? "failed" : "ok");
    return bad != 0;
}
