// Part of the two-pass lengths of fft_two.cuh (translation units of about equal
// compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part4(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<6, 4>(), two_pass_make<9, 6>(), two_pass_make<10, 9>(), two_pass_make<25, 5>(),
        two_pass_make<15, 12>(), two_pass_make<20, 15>(), two_pass_make<27, 20>(), two_pass_make<25, 25>(),
        two_pass_make<30, 27>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
