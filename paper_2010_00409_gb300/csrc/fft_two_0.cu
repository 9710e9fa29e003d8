// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part0(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<8, 4>(), two_pass_make<9, 5>(), two_pass_make<10, 10>(), two_pass_make<16, 10>(),
        two_pass_make<20, 10>(), two_pass_make<25, 15>(), two_pass_make<24, 16>(), two_pass_make<24, 24>(),
        two_pass_make<32, 30>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
