// How an LM-head call of the pair kernel is dealt out: columns of the MMAs, tiles cut into pieces, row blocks side by side.  Host code.
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
    double cost;        // rounds that the call takes
};
inline LmSlices plan_slices(int n_tiles, int pairs, int n_pad) {
    const int n_chunks = (n_pad + 31) / 32, rest = n_tiles % pairs;
    LmSlices r{n_tiles / pairs, 0, 0, 0.0};
    double best = rest > 0 ? 0.9 : 0.0;                // of a round
    for (int w = 1; w < n_chunks && w <= 8 && rest > 0; ++w) {      // 32 w <= 256: one MMA
        const int s = (n_chunks + w - 1) / w;
        const int each = (rest * s + pairs - 1) / pairs;
        const double cost = each * ((double)w / n_chunks + 0.25);
        if (cost < best) { best = cost; r.slices = s; r.slice_chunks = w; }
    }
    r.cost = r.rounds + (r.slices > 0 || rest == 0 ? best : 1.0);
    return r;
}

// Whether a row block of more than 256 rows and the one behind it share a launch, side by side: each has half of the pairs, and a
// tile of W that both come to at about the same time crosses HBM once (in launches one behind the other, twice).  That saves a
// launch and a merge, about 9 us, and wherever the halves' rounds add up to less than the whole's; but both blocks are
// multiplied with the columns of the first.  Estimated in columns of a round, one of which takes 3e-5 us per
// hidden dimension (0.106 us at 3584); a second block of at most 256 rows, whose epilogue hides behind the next tile,
// takes a sixth less alone.  Measured, one behind the other and side by side, us (at the power limit for the larger ones):
//   vocabulary 152064, hidden size 3584: 544 rows 585 556, 600 632 601, 800 763 743, 961 915 904, 513 (272 and 241 rows, 288 columns
//   and 256) 541 563, 577 (320 and 288) 632 618; 128256 and 4096: 600 rows 590 579, 513 512 562, 577 595 608, 769 717 756;
//   81920 (eight rounds and two thirds of one, or nine) 769 rows 393 402; 50257 and 2048: 513 rows 105 101, 960 169 146; 152064 and
//   1024: 513 rows 170 187; 4099 and 1024: 600 rows 21.1 12.1.
// Over 263 such calls this picks the slower way in 11, by 0.6 to 2.8 %.
inline bool side_by_side(int rows, int next_rows, int Hd, int n_tiles, int pairs) {
    if (pairs < 2 || next_rows < 1) return false;
    const double launch = 9.0 / 3e-5 / Hd;
    const LmColumns a = lm_columns(rows), b = lm_columns(next_rows);
    const double both = plan_slices(n_tiles, pairs / 2, a.padded()).cost * a.padded() + launch;
    const double alone = plan_slices(n_tiles, pairs, a.padded()).cost * a.padded() + launch;
    const double next = (b.n_parts == 2 ? plan_slices(n_tiles, pairs, b.padded()).cost : 0.84 * ((n_tiles + pairs - 1) / pairs)) * b.padded() + launch;
    return both <= 1.015 * (alone + next);
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
