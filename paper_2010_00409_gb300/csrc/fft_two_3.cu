// A quarter of the two-pass lengths of fft_two.cuh (translation units of about
// equal compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part3(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<6, 3>(), two_pass_make<6, 4>(), two_pass_make<8, 5>(), two_pass_make<10, 5>(),
        two_pass_make<10, 6>(), two_pass_make<10, 10>(), two_pass_make<15, 9>(), two_pass_make<15, 12>(),
        two_pass_make<16, 12>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
