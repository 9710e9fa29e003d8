// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part7(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<5, 5>(), two_pass_make<10, 6>(), two_pass_make<9, 9>(), two_pass_make<16, 12>(),
        two_pass_make<15, 15>(), two_pass_make<20, 18>(), two_pass_make<24, 18>(), two_pass_make<30, 24>(),
        two_pass_make<27, 27>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
