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
    // the rows of A there are to load and with the share of the SMs at work.  Fitted to 4685 products of 1-9000 rows,
    // 8-65536 columns and 32-14336 of K, both layouts, weights in L2 and not, every kernel timed on each: the choice costs
    // 1.1 % on average against the best of them.
    const long long slices = (K + 63) / 64;
    auto waves = [](long long tiles, long long slots) { return (tiles + slots - 1) / slots; };
    auto share = [&](long long ctas) { return ctas < sms ? double(ctas) / sms : 1.; };
    const double rows = M < 128 ? M / 128. : 1.;
    // Up to 128 rows the time goes into reading B from HBM; with a handful, all CTAs also fetch the same few lines of A at the
    // same time (14336 columns, K = 4096, one CTA per 128 x 128 tile: 16 to 128 rows 26-29 us, 8 rows or fewer 38-40).
    const double crowding = M > 128 ? 0. : M > 8 ? 0.1 : 0.3, crowding_wide = M > 128 ? 0.06 : M > 8 ? 0.08 : 0.1;
    const double ragged = (K % 64 || (b_nmajor && N % 64)) ? 1.1 : 1.;  // rows that do not begin on a 128-byte line
    GemmChoice g;
    // 128 x 256 tiles, one CTA each
    const long long tiles_wide = (long long)((M + 127) / 128) * ((N + 255) / 256);
    double best = 1.8 + waves(tiles_wide, sms) * (1.7 + slices * (0.34 + 0.07 * rows + crowding_wide * share(tiles_wide)));
    // CTA pairs move the fewest bytes per product (n = 4096: 96 us, against 105 us for 128 x 256 tiles of one CTA;
    // 8192 x 8192 x 4096: 351 / 425 us); a tile width that just fills the last wave saves up to a third of it
    // (420 x 6544 x 3840: 24.4 us 256 wide, 19.5 us 192 wide).  N-contiguous B comes in 64 columns per CTA at a time: 192 would
    // load as much as 256.  With at most 128 rows a pair's second CTA would have none.
    for (int w = 256; M > 128 && w >= 128; w -= b_nmajor ? 128 : 64) {
        const long long t = (long long)((M + 255) / 256) * ((N + w - 1) / w);
        const double cost = 3.5 + waves(t, sms / 2) * (1.6 * w / 256 + slices * (0.183 + (0.143 + 0.02 * share(2 * t)) * w / 256));
        if (cost < best) best = cost, g.tile_n = w;
    }
    // 128 x 128 tiles of one CTA each while each has an SM, or of a cluster that shares out K, which costs an exchange of the
    // sums.  (A cluster sits inside a GPC, so that not all SMs can be used by large ones: sixteen clusters of eight, or 35
    // of four, were not resident at once, and a second wave costs more than sharing K gains.)
    const long long tiles = (long long)((M + 127) / 128) * ((N + 127) / 128);
    for (int x = 1; x <= kGemmMaxSplits; x *= 2) {
        const long long resident = x == 8 ? 2 * sms / 3 : x == 4 ? 7 * sms / 8 : sms;
        if (x * tiles > resident || (x > 1 && x * 4 > slices)) break;
        const double cost = (x == 1 ? 3. : x == 2 ? 6.5 : x == 4 ? 6.4 : 7.3) +
                            (slices + x - 1) / x * (0.22 + 0.06 * rows + crowding * share(x * tiles)) * ragged;
        if (cost < best) best = cost, g.splits = x;
    }
    return g;
}

}  // namespace ave
