// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part5(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<9, 3>(), two_pass_make<8, 5>(), two_pass_make<12, 10>(), two_pass_make<16, 8>(),
        two_pass_make<18, 12>(), two_pass_make<20, 20>(), two_pass_make<27, 15>(), two_pass_make<27, 25>(),
        two_pass_make<32, 24>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
