// How many key chunks a launch of the 128-key attention kernel is cut into, and which launches are the 64-key kernel's.  Host code.
#pragma once
#include "attention_shared.cuh"

namespace sdv {

// The 128-key kernel (attention_wide.cu) runs one CTA per SM.  One round of it takes 5 us, or about 6 with a merge of
// chunks, plus 0.02 us per CTA (they share the memory that the first copies come from), plus 0.4 us per cache block
// of its longest chunk, in tiles of two, plus about 0.5 us where the next call's CTAs find no free SMs to set up on
// while this one runs: fitted to calls of 1 to 16 sequences of 200 to 8192 tokens, trees of 11, 28 and 60 nodes, 1 to 8
// chunks, of which it picks one within 1.5 % of the fastest on average (12 % at most).  With 8 us and 2.8 to 3.8 us for
// the merge, which it took before, middling sequences stayed whole or in two for too long: two of 900 tokens and 60 nodes
// 11.2 us instead of 10.0, four of 1100 13.0 instead of 11.7, eight of 1300 and 28 nodes 14.4 instead of 12.8.  In
// launches of several rounds, where nothing overlaps a round's ends, each takes 11 us, the merge, and 0.36 us per block.
// Measured per call in us for 1 to 8 chunks: one sequence of 2048 tokens and 60 nodes 16.4 12.7 10.9 9.9 9.9 10.1 15.6
// 15.2 (16 clusters of seven or eight are more than fit at a time), of 8192 50.8 29.7 22.1 18.3 17.1 16.0 25.1 23.7, one
// chain of 11 nodes over 4096 27.8 18.0 14.3 12.2 11.5 11.0 10.5 9.9.  Chunk counts that are no powers of two fill SMs that
// those leave idle: ten such
// chains 19.3 us with three chunks (21.4 with two), five sequences of 2000 tokens with 16 heads 13.0 (14.6).
// The table's width stands for the longest length here, which the host does not know: a table that is far wider
// makes long launches look longer than they are (in a table of 512 blocks 256 CTAs of 1000 tokens take 26.4 instead
// of 22.7 us, 160 of 2048 54.6 instead of 35), but what a single round's sequences are cut into follows from
// their own lengths.
// Where one round has room for every row tile, several are taken only if they take at least a fifth off the blocks that
// an SM works through (rounds / chunks against 1 / chunks of the one round), as three chunks in two rounds do for 80 row tiles
// (five sequences of 8192 tokens 46.8 instead of 55 us, of 28000 135 instead of 176) and four in three for 96 (28000
// tokens 160 instead of 174).  Otherwise they only repeat a round's ends, and the table's width alone must not bring them about:
// the two estimates' slopes differ, so that from 434 blocks on 128 row tiles went in two rounds of pairs, eight
// sequences of 1000 tokens and 60 nodes 22.3 us instead of 13.4 in a table of 512, of 4096 39.3 instead of 31.4.  So did 64
// row tiles from 831 blocks on, in two rounds of four chunks (four sequences of 1000 tokens in 2048 blocks 19.5 instead
// of 11.3), and 40 in two of six instead of one of three (ten chains of 4096 there 28.2 instead of 19.1).  A saving of
// a seventh is none: ten chains of 28000 in two rounds of seven chunks 120 us, in one of three 92.
// The 64-key kernel's two CTAs per SM overlap each other's ends: a round of twice as many CTAs takes about
// 0.9 us per block plus 13 us.  It is left for launches of several rounds in which those ends weigh more
// (256 CTAs of 1000 tokens: 28.7 against 33.9 us; of 4096: 71.4 against 69.9; 1792 CTAs of 4096 tokens under the
// power cap, where 64-key tiles cost more energy: 569 against 544).
//
// base: row tiles of the launch (layers x sequences x KV heads x row tiles of a sequence); blocks: width of the block table;
// forced_chunks: test hook (0: none); resident(c): how many clusters of c CTAs run at a time.  Sets n_chunks and how a
// sequence is cut.  false: the 64-key kernel is faster.
template <class Resident>
inline bool choose_wide(AttnPlan* p, long long base, int blocks, int sms, int forced_chunks, Resident resident) {
    const double merge[kMaxChunks] = {0.0, 2.8, 3.2, 3.2, 3.3, 3.4, 3.6, 3.8};
    int n = 1;
    long long n_rounds = 1;
    double best = 1e30;
    int one_round = 0;                                     // the most chunks that one round has room for
    p->tree_blocks = kTreeBlocks;
    const bool forced = forced_chunks > 0 && forced_chunks <= blocks;
    auto whole = [&](int c) { return forced ? 0 : (c == 2 ? 10 : 5); };   // blocks of a sequence that is not cut, see below
    for (int c = 1; c <= kMaxChunks && c <= blocks; ++c) {
        const long long rounds = (base + resident(c) - 1) / resident(c);
        if (rounds == 1) one_round = c;
        if (c > 1 && blocks <= whole(c)) continue;         // (CTAs without work: eight chains of 200 tokens 7.6 instead of 7.0 us)
        if (!forced && rounds > 1 && 5 * rounds * one_round > 4 * c) continue;
        double us = rounds * (11.0 + merge[c - 1] + 0.36 * ((blocks + c - 1) / c));
        if (rounds == 1) {                                 // blocks of the longest chunk, of a sequence and its tree that fill the table
            p->set_chunks(c, whole(c));
            const ChunkRange last = chunk_range(*p, ((blocks < (1 << 24) ? blocks : 1 << 24) - 1) * kBlock, blocks, c - 1);
            const int per = last.tpc > last.t1 - last.t0 ? last.tpc : last.t1 - last.t0 + 1;
            us = (c == 1 ? 5.0 : 5.8 + 0.1 * c) + 0.02 * base * c + (2 * base * c > sms ? 0.52 : 0.0) + 0.28 * per + 0.25 * ((per + 1) / 2);
        }
        if (forced ? c == forced_chunks : us < best - 1e-9) { best = us; n = c; n_rounds = rounds; }
    }
    if (n_rounds > 1) {
        const double rounds = base <= 2 * sms ? 1.0 : (double)base / (2 * sms) + 0.25;     // a partial round, cut into chunks
        if (best > 1.05 * rounds * (13.0 + 0.9 * blocks)) return false;
    }
    // Where all clusters run at once, a sequence so short that the merge costs more than the split saves stays whole
    // (us per call uncut, in two, three, four, six chunks, one sequence and 60 nodes: 4 blocks 7.1 7.6 7.6 7.6, 6 blocks
    // 8.1 8.2 8.1 7.9 7.9, 8 blocks 8.6 8.6 8.0 7.9 7.7, 12 blocks 10.0 9.5 9.0 9.0 8.1); the others are cut as far as the
    // cluster goes.  This must not follow from the table's width, of which a chunk's size was once a share: then one
    // sequence of 2048 tokens in a table of 512 blocks ran whole (16.3 us, now 9.8; 10.2 in a table of 33), eight chains
    // of 4096 took 28.7 (17.0), one of 8192 in 2048 blocks 50.7 (16.0).  The other side: in a batch of very different
    // lengths the short sequences take memory bandwidth from the longest (eight chains over 200 to 8192 tokens
    // 20.4 us, 19.8 with chunks as long as the longest's; 100 to 3000 tokens 11.4 against 11.7).
    // In several rounds every sequence is cut alike: the CTAs that leave would still hold back the next cluster
    // (half-empty pairs halved the machine).
    p->set_chunks(n, n_rounds > 1 ? -1 : whole(n));
    return true;
}

// Whether the 128-key kernel's first copies go first.  Calls of several rounds keep the other order: nothing waits for their
// later CTAs' copies (72 chains of 1000 tokens, eight calls 248.1 248.7; 256 row tiles of one sequence of 4000 545 561).  In one round
// latencies count, 1 to 3 % of the calls below, but a row tile's loop takes 40 to 80 of 1270 cycles a tile longer, which shows
// where several row tiles share K and V: the line is the blocks of a chunk, fitted for each number of chunks.  Fourteen calls in a row,
// us, without and with, sequences of 60 nodes and their blocks a chunk: one chunk, eight of 1250 (20) 204.0 203.6, 1300
// (22) 206.0 204.8, 1350 (23) 214.3 215.9, six of 1500 (25) 222.7 225.9; two chunks, four of 2100 (17) 195.8 193.9, 2200 (18) 201.8
// 204.3, 2700 (22) 222.6 227.8, three of 2200 (18) 1.3 % longer; three chunks, two of 1000 (6) 1.1 % shorter, three of 2500 (14) 214.1
// 215.9, 4000 (22) 274.4 281.0; four, two of 5500 (22) 224.4 222.2, 6500 (26) 243.5 242.5; six, one of 8192 (22) 1.2 % shorter, 12000 (32)
// 0.4 % longer.  With one or two row tiles the line may be anywhere from 22 up (four sequences of 28 nodes and 2900 tokens 2.2 %
// shorter, eight of 2700 in two chunks of 22 233.1 233.9); chains, one row tile, gain at every length (eight of 10000 1 %).
// The blocks are the table's width, which stands for the longest length as above: in a table that is far wider a call keeps the
// order that is right for long sequences and misses the gain (28 calls, one sequence of 2048 tokens in 33 blocks 269, in 512 275).
inline bool copies_first(const AttnPlan& p, int blocks) {
    constexpr int kLine = 22, kLineShared[kMaxChunks] = {kLine, 17, 12, kLine, kLine, kLine, kLine, kLine};
    if (p.whole_blocks < 0) return false;                  // several rounds
    const int per = (blocks + p.n_chunks - 1) / p.n_chunks;
    return p.row_tiles == 1 || per <= (p.row_tiles == 2 ? kLine : kLineShared[p.n_chunks - 1]);
}

}  // namespace sdv
