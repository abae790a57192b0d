// How an LM-head call of the pair kernel is dealt out: columns of the MMAs, tiles cut into pieces.  Host code.
#pragma once

namespace sdv {

// The hidden rows of a block as MMA columns: one or two MMAs along N per k-step, part_n (a multiple of 16, at most 256) each.
struct LmColumns {
    int n_parts, part_n;
    int padded() const { return n_parts * part_n; }
};
inline LmColumns lm_columns(int rows) {
    const int n16 = (rows + 15) / 16 * 16, parts = n16 > 256 ? 2 : 1;
    return {parts, ((n16 + parts - 1) / parts + 15) / 16 * 16};
}

// More than 256 hidden rows, where the tensor cores bound a tile: if few tiles are left over after whole rounds of
// all pairs (or there are few tiles at all), they are cut along the hidden rows into pieces that are dealt out to
// all pairs.  A piece costs its share of a tile and about a quarter more: it streams its tile's W through the
// pair once again, and fills and drains the pipeline.  480 rows, hidden size 3584: vocabulary of 4099 39.1 -> 24.7 us,
// 152064 (594 tiles, 74 pairs) 377 -> 368; cutting the 49 tiles left over at 50257 took 82 instead of 78, and up to
// 256 rows, where streaming W is what takes the time, pieces are as slow as whole tiles.
struct LmSlices {
    int rounds;         // whole rounds, if the rest is cut
    int slices;         // pieces of a tile of the rest, 0: none is cut
    int slice_chunks;   // 32-row chunks of a piece
};
inline LmSlices plan_slices(int n_tiles, int pairs, int n_pad) {
    const int n_chunks = (n_pad + 31) / 32, rest = n_tiles % pairs;
    LmSlices r{n_tiles / pairs, 0, 0};
    double best = 0.9;                                 // of a round
    for (int w = 1; w < n_chunks && w <= 8 && rest > 0; ++w) {      // 32 w <= 256: one MMA
        const int s = (n_chunks + w - 1) / w;
        const int each = (rest * s + pairs - 1) / pairs;
        const double cost = each * ((double)w / n_chunks + 0.25);
        if (cost < best) { best = cost; r.slices = s; r.slice_chunks = w; }
    }
    return r;
}

// Whether a CTA has the first eight k-steps of 64 of its first tile of W brought to L2 while the kernel ahead runs.  Calls in a row, W from HBM, us without
// and with: 60 rows, hidden size 4096 and vocabulary of 32000 47.1 45.3, 2048 and 50257 37.8 36.2, 768 and 32000 14.4 13.1; chains'
// tail at 3584 and 152064 208.8 208.2; 480 rows, 1024 and 1025 10.9 10.6; three k-steps give half of that.  Not where a CTA has no
// second tile and eight k-steps are much or all of the one it has, which its copies ask for at once anyway: 60 rows, 512 and 6000
// 7.2 7.6, 4099 7.0 7.4; 384 and 6000 6.9 7.2; 480 rows, 256 and 6000 9.3 9.7.  (A hidden size of 128 has so little W that it gains
// again: 60 rows and 6000 6.0 5.9.)
constexpr int kAheadSteps = 8;
inline bool brings_ahead(int Hd, int n_tiles, int pairs) { return Hd < 256 || Hd >= 1024 || n_tiles >= pairs; }

}  // namespace sdv
