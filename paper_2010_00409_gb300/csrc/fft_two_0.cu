// A quarter of the two-pass lengths of fft_two.cuh (translation units of about
// equal compile time).
#include "fft_two.cuh"

namespace psatd {

const TwoPassEntry* two_pass_part0(int N) {
    static const TwoPassEntry entries[] = {
        two_pass_make<9, 3>(), two_pass_make<6, 6>(), two_pass_make<9, 6>(), two_pass_make<9, 8>(),
        two_pass_make<10, 9>(), two_pass_make<16, 8>(), two_pass_make<12, 12>(), two_pass_make<16, 16>()};
    for (const TwoPassEntry& e : entries)
        if (e.N == N) return &e;
    return nullptr;
}

}  // namespace psatd
