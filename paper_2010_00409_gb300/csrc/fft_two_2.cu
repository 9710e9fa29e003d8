// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part2(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<6, 3>(), two_pass_make<8, 8>(), two_pass_make<15, 5>(), two_pass_make<15, 10>(),
        two_pass_make<16, 16>(), two_pass_make<20, 16>(), two_pass_make<24, 20>(), two_pass_make<25, 24>(),
        two_pass_make<32, 27>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
