// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part6(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<5, 4>(), two_pass_make<9, 8>(), two_pass_make<10, 8>(), two_pass_make<18, 9>(),
        two_pass_make<16, 15>(), two_pass_make<18, 18>(), two_pass_make<27, 18>(), two_pass_make<32, 20>(),
        two_pass_make<30, 25>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
