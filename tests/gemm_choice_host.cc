// Host build of the choice between the matrix-product kernels, for the unit tests: the library's own header
// (paper_2604_18616_b200/csrc/gemm_choice.cuh) behind a flat C interface.
#include "../paper_2604_18616_b200/csrc/gemm_choice.cuh"

// splits > 0: clusters of that many CTAs; 0: 128 x 256 tiles; < 0: CTA pairs, minus the tile's columns.
extern "C" int gc_choose(int b_nmajor, int M, int N, int K, int sms) {
    const ave::GemmChoice g = ave::choose_gemm(b_nmajor != 0, M, N, K, sms);
    return g.splits > 0 ? g.splits : -g.tile_n;
}
