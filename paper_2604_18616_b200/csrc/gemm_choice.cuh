// Which of the matrix-product kernels a product runs.  No CUDA types, so that unit tests compile it for the host.
#pragma once

namespace ave {

constexpr int kGemmMaxSplits = 8;  // CTAs of a cluster that share a tile's K

struct GemmChoice {
    int splits = 0;  // > 0: 128 x 128 tiles of a cluster of this many CTAs (one: a CTA each)
    int tile_n = 0;  // else > 0: CTA pairs with tiles of 256 x tile_n; else 128 x 256 tiles of one CTA each
};

// C[M, N], a reduction over K, on a part with `sms` SMs; b_nmajor: B is [K, N].
inline GemmChoice choose_gemm(bool b_nmajor, int M, int N, int K, int sms) {
    // Each kernel's time in us: a constant, and per wave of tiles a constant and a time per slice of 64 of K, which grows with
    // the rows of A and the columns of B that there are to load, and with few rows also with the share of the SMs at work.
    // Fitted to 9388 products of 1-9000 rows, 8-64000 columns and 32-14400 of K, both layouts, weights in L2 and not, every
    // kernel timed on each: the choice costs 0.7 % on average against the best of them.
    const long long slices = (K + 63) / 64;
    auto waves = [](long long tiles, long long slots) { return (tiles + slots - 1) / slots; };
    auto share = [&](long long ctas) { return ctas < sms ? double(ctas) / sms : 1.; };
    auto part = [](int size, int of) { return size < of ? double(size) / of : 1.; };  // of a tile's rows or columns
    const double rows = part(M, 128);
    // Up to 128 rows the time goes into reading B from HBM; with a handful, all CTAs also fetch the same few lines of A at the
    // same time (14336 columns, K = 4096, one CTA per 128 x 128 tile: 16 to 128 rows 26-29 us, 8 rows or fewer 38-40).
    const double crowding = M > 128 ? 0. : M > 8 ? 0.055 : 0.37, crowding_wide = M > 128 || M <= 8 ? 0.06 : 0.08;
    const bool ragged = K % 64 || (b_nmajor && N % 64);  // rows that do not begin on a 128-byte line
    GemmChoice g;
    // 128 x 256 tiles, one CTA each
    const long long tiles_wide = (long long)((M + 127) / 128) * ((N + 255) / 256);
    double best = 1.63 + waves(tiles_wide, sms) *
                             (1.78 + slices * (0.269 + 0.08 * rows + 0.063 * part(N, 256) + crowding_wide * share(tiles_wide)) *
                                         (ragged ? 1.21 : 1.));
    // CTA pairs move the fewest bytes per product (n = 4096: 96 us, against 105 us for 128 x 256 tiles of one CTA;
    // 8192 x 8192 x 4096: 351 / 425 us); a tile width that just fills the last wave saves up to a third of it
    // (420 x 6544 x 3840: 24.4 us 256 wide, 19.5 us 192 wide).  N-contiguous B comes in 64 columns per CTA at a time: 192 would
    // load as much as 256, 64 as much as 128.  With at most 128 rows a pair's second CTA would have none.
    for (int w = 256; M > 128 && w >= (b_nmajor ? 128 : 64); w -= b_nmajor ? 128 : 64) {
        const double cost = 3.31 + waves((long long)((M + 255) / 256) * ((N + w - 1) / w), sms / 2) *
                                       (1.5 * w / 256 + slices * (0.192 + 0.162 * part(N, w) * w / 256));
        if (cost < best) best = cost, g.tile_n = w;
    }
    // 128 x 128 tiles of one CTA each while each has an SM, or of a cluster that shares out K, which costs an exchange of the
    // sums.  (A cluster sits inside a GPC, so that not all SMs can be used by large ones: sixteen clusters of eight, or 35
    // of four, were not resident at once, and a second wave costs more than sharing K gains.)
    const long long tiles = (long long)((M + 127) / 128) * ((N + 127) / 128);
    for (int x = 1; x <= kGemmMaxSplits; x *= 2) {
        const long long resident = x == 8 ? 2 * sms / 3 : x == 4 ? 7 * sms / 8 : sms;
        if (x * tiles > resident || (x > 1 && x * 4 > slices)) break;
        const double cost = (x == 1 ? 2.88 : x == 2 ? 6.2 : x == 4 ? 6.36 : 6.1) +
                            (slices + x - 1) / x * (0.179 + 0.06 * rows + 0.04 * part(N, 128) + crowding * share(x * tiles)) *
                                (ragged ? 1.125 : 1.);
        if (cost < best) best = cost, g.splits = x;
    }
    return g;
}

}  // namespace ave
