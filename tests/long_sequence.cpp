// The resident time loops count steps in 32 bits: a longer sequence is left to the path that issues steps one by one
// (return value 1, before anything is planned).  Prints the return value for one step more than they take.
#include <cstdio>

#include "../paper_2005_05758_b200/csrc/csb_rnn1.hpp"

int main() {
    csb_matrix A;
    const csb_matrix* W[1] = {&A};
    const int in = 1;
    const float x = 0.f;
    std::printf("%d\n", csb::rnn1_forward(csb::kR1Ligru, 1, W, nullptr, nullptr, &x, 1ll << 31, 1, 1, 1, &in, nullptr, nullptr, nullptr, nullptr, nullptr, 0u, nullptr));
    return 0;
}
