// Runs one host-side piece of the library with every allocation failing from the n-th on, in whichever thread it comes.
// Exit code 0: it returned a status (or, planners, threw std::bad_alloc to their caller); an abort has another.
#include <atomic>
#include <cstdlib>
#include <new>

#include "../paper_2005_05758_b200/csrc/csb_rnn1.hpp"
#include "../paper_2005_05758_b200/csrc/csb_rnn_unit.hpp"

static std::atomic<long> g_left{-1};                       // allocations that still succeed; < 0: all
static void* take(size_t n) {
    long left = g_left.load();
    while (left > 0 && !g_left.compare_exchange_weak(left, left - 1)) {}
    void* p = left == 0 ? nullptr : std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void* operator new(size_t n) { return take(n); }
void* operator new[](size_t n) { return take(n); }
void* operator new(size_t n, const std::nothrow_t&) noexcept { try { return take(n); } catch (...) { return nullptr; } }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
void operator delete[](void* p, size_t) noexcept { std::free(p); }

using namespace csb;

int main(int argc, char** argv) {
    if (argc < 3) return 2;
    const int R = 2048, C = 1024, b = 32, I = C - R / 4;
    unsigned int state = 1;
    auto draw = [&]() { return (state = state * 1664525u + 1013904223u) >> 16; };
    std::vector<float> W((size_t)R * C);
    std::vector<uint8_t> rk((size_t)R * C / b), ck(rk.size());
    for (float& w : W) w = (float)(draw() % 1000) / 1000.f;
    for (uint8_t& k : rk) k = draw() & 1;
    for (uint8_t& k : ck) k = draw() & 1;
    csb_matrix* A = nullptr;
    csb_matrix* Z = nullptr;
    if (csb_encode(W.data(), R, C, C, b, b, rk.data(), ck.data(), CSB_F16, -1, nullptr, &A) != CSB_OK) return 3;
    const csb_matrix* M[1] = {A};
    int64_t info[8];
    int rc = CSB_OK;
    g_left = std::atol(argv[2]);
    switch (std::atoi(argv[1])) {
        case 0: rc = csb_encode(W.data(), R, C, C, b, b, rk.data(), ck.data(), CSB_F32, -1, nullptr, &Z); break;
        case 1: rc = csb_plan_dump(A, 148, 16, 4096, info, nullptr, 0, nullptr, 0, nullptr, 0); break;
        case 2: rc = csb_panel_dump(A, 148, 32, 16384, info, nullptr, 0, nullptr, 0); break;
        case 3: rc = csb_spmm_plan_dump(A, 32, 148, info, nullptr, 0, nullptr, 0, nullptr, 0, nullptr, 0); break;
        case 4: { RuHostPlan P; try { rc = plan_unit_host(kR1Lstm, 1, M, nullptr, &I, R / 4, R / 4, 1, 64, &P); } catch (const std::bad_alloc&) { rc = CSB_ERR_ALLOC; } break; }
        default: { R1HostPlan P; try { rc = plan_rnn1_host(kR1Lstm, 1, M, nullptr, &I, R / 4, R / 4, 1, 64, (size_t)1 << 40, &P); } catch (const std::bad_alloc&) { rc = CSB_ERR_ALLOC; } break; }
    }
    g_left = -1;
    return rc == CSB_OK || rc == CSB_ERR_ALLOC ? 0 : 4;
}
