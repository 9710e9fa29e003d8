// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part1(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<6, 6>(), two_pass_make<8, 6>(), two_pass_make<12, 9>(), two_pass_make<15, 9>(),
        two_pass_make<25, 10>(), two_pass_make<18, 15>(), two_pass_make<25, 20>(), two_pass_make<32, 16>(),
        two_pass_make<30, 30>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
