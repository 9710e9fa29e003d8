// A quarter of the two-pass lengths of fft_two.cuh (translation units of about
// equal compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part1(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<5, 4>(), two_pass_make<5, 5>(), two_pass_make<9, 5>(), two_pass_make<8, 6>(),
        two_pass_make<9, 9>(), two_pass_make<12, 8>(), two_pass_make<12, 10>(), two_pass_make<15, 10>(),
        two_pass_make<16, 15>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
