// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part3(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<6, 5>(), two_pass_make<10, 5>(), two_pass_make<12, 8>(), two_pass_make<12, 12>(),
        two_pass_make<27, 9>(), two_pass_make<18, 16>(), two_pass_make<25, 18>(), two_pass_make<27, 24>(),
        two_pass_make<32, 25>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
