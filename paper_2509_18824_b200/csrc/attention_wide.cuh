// Pieces of the 128-key attention kernels: shared-memory layout, and the softmax of a CTA's tiles.
#pragma once
#include <type_traits>
#include "attention_shared.cuh"

namespace sdv {

constexpr int kWTile = 128;                     // keys per tile: two cache blocks
constexpr int kWThreads = 320;                  // warps 0-3, 4-7 softmax groups, warp 8 TMA, warp 9 MMA issuer
constexpr int kWTmaWarp = 8, kWMmaWarp = 9;
constexpr int kWStages = 3;                     // K and V ring slots, score buffers
constexpr int kWHalf = kWTile * 128;            // bytes of one D-half of a tile: [128 keys][64] bf16, swizzled (16 KiB)
constexpr int kWStage = 2 * kWHalf;             // 32 KiB
constexpr int kWQBytes = 2 * kRowTile * 128;    // 32 KiB
constexpr int kWBars = 256;                     // barriers and two words
constexpr int kWSmem = kWQBytes + 2 * kWStages * kWStage + kWBars + 3 * kRowTile * 4;   // + references, two groups' sums

// Where everything lives in the dynamic shared memory.
struct WideShared {
    uint8_t *q_smem, *k_smem, *v_smem;
    uint64_t* k_full;       // [3] TMA -> MMA
    uint64_t* v_full;       // [3] TMA -> MMA (and whoever clears V rows)
    uint64_t* s_full;       // [3] MMA -> softmax, TMA: scores of tile j in buffer j % 3, K slot j % 3 read
    uint64_t* v_empty;      // [3] MMA -> TMA: O updated by tile j, V slot j % 3 read
    uint64_t* p_full;       // [3] softmax -> MMA: P of tile j written over its scores
    uint64_t* commit;       // [4] per TMEM quadrant: tile j's softmax is final (phase j)
    uint64_t* ref_full;     // [4] per TMEM quadrant: the first tile's reference is known
    uint64_t* o_full;       // MMA -> softmax: every MMA of a row tile has completed
    uint64_t* q_full;       // TMA -> MMA
    uint64_t* x_full;       // the other chunks' rows have arrived
    uint32_t* tmem_slot;
    int* abort_flag;
    int* seq;               // sequence_of_rank
    float* ref_smem;        // [128] by TMEM lane
    float* sum_smem;        // [2][128]

    __device__ __forceinline__ explicit WideShared(uint8_t* smem) {
        q_smem = smem;
        k_smem = smem + kWQBytes;
        v_smem = k_smem + kWStages * kWStage;
        uint64_t* bars = reinterpret_cast<uint64_t*>(v_smem + kWStages * kWStage);
        k_full = bars; v_full = bars + 3; s_full = bars + 6; v_empty = bars + 9; p_full = bars + 12; commit = bars + 15;
        o_full = bars + 19; q_full = bars + 20; x_full = bars + 21; ref_full = bars + 22;
        tmem_slot = reinterpret_cast<uint32_t*>(bars + 26);
        abort_flag = reinterpret_cast<int*>(bars + 27);
        seq = reinterpret_cast<int*>(bars + 28);
        ref_smem = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kWBars);
        sum_smem = ref_smem + kRowTile;
    }
    // (one thread)
    __device__ __forceinline__ void init_barriers() const {
        *abort_flag = 0;
        for (int i = 0; i < kWStages; ++i) {
            mbar_init(&k_full[i], 1); mbar_init(&v_full[i], 1); mbar_init(&s_full[i], 1);
            mbar_init(&v_empty[i], 1); mbar_init(&p_full[i], 4);
        }
        for (int i = 0; i < 4; ++i) { mbar_init(&commit[i], 1); mbar_init(&ref_full[i], 1); }
        mbar_init(o_full, 1); mbar_init(q_full, 1); mbar_init(x_full, 1);
    }
};

// What a CTA has to do for a sequence of len cached tokens and n nodes: its share of the key chunks.
struct WideWork {
    int n, len;
    int n_chunks;                   // key chunks of this sequence
    int tiles_total, tpc;           // cache blocks of the sequence and of a chunk, see chunk_range
    int t0, n_pref;                 // this chunk's first cache block, and how many
    int nb;                         // blocks of keys: those, and the tree's in the last chunk
    // (what has been worked out stays in front of the code that follows)
    __device__ __forceinline__ void settle() {
        asm volatile("" : "+r"(n), "+r"(len), "+r"(n_chunks), "+r"(tiles_total), "+r"(tpc), "+r"(t0), "+r"(n_pref), "+r"(nb));
    }
};
__device__ __forceinline__ WideWork wide_work(const sd_batch& bt, const AttnPlan& plan, int n, int len, int chunk) {
    WideWork w;
    w.n = min(max(n, 0), bt.T_max);
    w.len = min(max(len, 0), 0x7fffffff - kBlock);         // (any number may stand there before the kernel ahead is done)
    const ChunkRange cr = chunk_range(plan, w.len, bt.max_blocks_per_seq, chunk);
    w.n_chunks = cr.n_chunks;
    w.tiles_total = cr.tiles_total;
    w.tpc = cr.tpc;
    w.t0 = cr.t0;
    w.n_pref = cr.t1 - cr.t0;
    w.nb = w.n_pref + (chunk == w.n_chunks - 1 ? 1 : 0);
    return w;
}

// The key tiles of one row tile: nt tiles over nb blocks, of which n_pref are cache blocks t0 .. of the sequence
// (len cached tokens, n nodes), the one behind them the tree's.
struct WideTiles { int nt, nb, n_pref, t0, len, n; };

// Softmax of those tiles by the two groups of four warps, one thread per row and group; false: a wait ran out.
__device__ __forceinline__ bool wide_softmax(const AttnPlan& plan, const WideShared& sh, const WideTiles& w, uint32_t tmem_o, uint32_t tmem_s,
                                             int group, int quad, int lane, bool row_ok, uint64_t amask, float scale_log2,
                                             float& m_used, float& l) {
    const int gt = quad * 32 + lane;
    const uint32_t lane_field = (uint32_t)(quad * 32) << 16;
    volatile float* my_ref = sh.ref_smem + gt;
    const uint64_t scale2 = pack_f32x2(scale_log2, scale_log2);
    uint64_t neg_m2 = 0ull;                            // -(reference of this row), twice
    const int n_full = max(min(w.len / kBlock - w.t0, w.n_pref), 0) / 2;   // leading tiles with all 128 keys inside the prefix
    // Loads, exponentials and stores of one tile against the row's reference (tile 0 sets it), see
    // exp_pack and kSumLimit.  0: done, 1: the reference has to be raised first (nothing stored yet), -1: a wait ran
    // out.  The usual tile has all keys visible; masked ones (the last: cache slots behind len, the tree's keys)
    // take the same body with the scores of hidden keys replaced.  (As a body of their own that looked for the
    // maximum first they took 4800 instead of 1500 cycles, at the end of every call.)
    auto tile = [&](auto masked, auto only_half, int j, const uint32_t (&mask)[4]) -> int {
        constexpr bool kMasked = decltype(masked)::value, half = decltype(only_half)::value;     // half: 64 keys
        const int s = j % kWStages;
        const uint32_t ts = tmem_s + lane_field + s * kWTile;
        if (j == 0) {
            // The reference: the largest of the first sixteen scores (any score of the row will do, see kSumLimit; a
            // maximum over all of them took 800 cycles in front of every call's first exponentials), or, where some
            // row sees none of those keys, of all.
            uint32_t a[16];
            tmem_ld16(ts, a);
            tmem_ld_wait();
            if (kMasked) mask_scores(a, mask[0]);
            float mt = fmaxf(__uint_as_float(a[0]), __uint_as_float(a[1]));
#pragma unroll
            for (int k = 2; k < 16; k += 2) mt = max3(mt, __uint_as_float(a[k]), __uint_as_float(a[k + 1]));
            if (kMasked && __any_sync(0xffffffffu, row_ok && mt == -INFINITY)) {
#pragma unroll 1
                for (int c = 0; c < (half ? 4 : 8); ++c) {
                    tmem_ld16(ts + c * 16, a);
                    tmem_ld_wait();
                    mask_scores(a, (c < 4 ? (c < 2 ? mask[0] : mask[1]) : (c < 6 ? mask[2] : mask[3])) >> ((c & 1) * 16));
#pragma unroll
                    for (int k = 0; k < 16; k += 2) mt = max3(mt, __uint_as_float(a[k]), __uint_as_float(a[k + 1]));
                }
            }
            m_used = row_ok ? mt * scale_log2 : 0.f;       // scale > 0; finite for rows that nobody reads
            *my_ref = m_used;
            neg_m2 = pack_f32x2(-m_used, -m_used);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.ref_full[quad]);   // (the other group need not wait for the tile)
        }
        uint32_t ra[16], rb[16], pk0[32], pk1[32];
        uint64_t ps[2] = {0ull, 0ull};
        tmem_ld16(ts, ra);                         // sixteen scores at a time, the next ones on their way
#pragma unroll
        for (int c = 0; c < 8; c += 2) {           // (thirty-two at a time left too few registers: spills)
            if (c == 4 && half) break;
            uint32_t* pk = (c < 4 ? pk0 : pk1) + (c & 2) * 8;
            tmem_ld_wait();
            tmem_ld16(ts + (c + 1) * 16, rb);
            if (kMasked) mask_scores(ra, mask[c / 2]);
            exp_pack(ra, scale2, neg_m2, pk, ps);
            tmem_ld_wait();
            if (c < 6 && !(c == 2 && half)) tmem_ld16(ts + (c + 2) * 16, ra);
            if (kMasked) mask_scores(rb, mask[c / 2] >> 16);
            exp_pack(rb, scale2, neg_m2, pk + 8, ps);
        }
        const float psum = sum_f32x2(add_f32x2(ps[0], ps[1]));
        // the tile before is final, and its reference still the one used here
        if (j > 0 && !mbar_wait(&sh.commit[quad], (uint32_t)(j - 1) & 1u, sh.abort_flag, plan.wait_cycles)) return -1;
        const float ref = *my_ref;
        if (__any_sync(0xffffffffu, row_ok && (!(psum <= kSumLimit) || ref != m_used))) return 1;
        l += psum;
        tmem_st32(ts, pk0);                        // P over the scores this thread has just consumed
        if (!half) tmem_st32(ts + 32, pk1);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0 && !(plan.withhold && j == 0)) { mbar_arrive(&sh.p_full[s]); mbar_arrive(&sh.commit[quad]); }
        return 0;
    };
    for (int j = group; j < w.nt; j += 2) {
        const int s = j % kWStages;
        const uint32_t ph = (uint32_t)(j / kWStages) & 1u;
        const uint32_t ts = tmem_s + lane_field + s * kWTile;
        if (j == 1) {                                      // the reference that the other group found in tile 0
            if (!mbar_wait(&sh.ref_full[quad], 0, sh.abort_flag, plan.wait_cycles)) return false;
            m_used = *my_ref;
            neg_m2 = pack_f32x2(-m_used, -m_used);
        }
        uint32_t mask[4] = {~0u, ~0u, ~0u, ~0u};           // visible keys of the four 32-key quarters
        if (!mbar_wait(&sh.s_full[s], ph, sh.abort_flag, plan.wait_cycles)) return false;
        tc_fence_after_sync();
        int done;
        if (j < n_full) {
            done = tile(std::false_type{}, std::false_type{}, j, mask);
        } else {
            // First the V rows of keys that no row may see (cache slots at and beyond len, rows of unused tree
            // nodes): they carry weight 0, but 0 x NaN or 0 x Inf would still poison the accumulator, so they are
            // cleared in shared memory before P.V reads them (the arrival on p_full orders the two).  This
            // comes after the wait for the scores of tile j: they were issued behind P.V of tile j - 3, which
            // read the V tile that used this ring slot before, so the slot's barrier is by now in the
            // phase of tile j.
            int v_rows[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = 2 * j + h;
                const bool tree = i >= w.n_pref;
                const int valid = i >= w.nb ? 0 : (tree ? kBlock : max(min(w.len - (w.t0 + i) * kBlock, kBlock), 0));
                v_rows[h] = i >= w.nb ? kBlock : (tree ? w.n : valid);
                const uint64_t m = (tree && i < w.nb) ? amask : (valid >= 64 ? ~0ull : ((1ull << valid) - 1ull));
                mask[2 * h] = (uint32_t)m; mask[2 * h + 1] = (uint32_t)(m >> 32);
            }
            if (v_rows[0] < kBlock || v_rows[1] < kBlock) {
                if (!mbar_wait(&sh.v_full[s], ph, sh.abort_flag, plan.wait_cycles)) return false;
                const int h = gt >> 6, key = gt & 63;
                if (key >= v_rows[h]) {
                    uint4* z = reinterpret_cast<uint4*>(sh.v_smem + s * kWStage + gt * 128);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        z[c] = make_uint4(0, 0, 0, 0);
                        z[c + kWHalf / 16] = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();
                }
            }
            done = 2 * j + 1 < w.nb ? tile(std::true_type{}, std::false_type{}, j, mask) : tile(std::true_type{}, std::true_type{}, j, mask);
        }
        if (done < 0) return false;
        if (done == 0) continue;
        // A score far above the reference (or one that is not a number), or the other group has raised the reference
        // since: the tile before is final by now; the reference is raised if need be and the tile redone.
        {
            const float ref = *my_ref;
            if (ref != m_used) { l *= exp2f(m_used - ref); m_used = ref; }
        }
        float mt = -INFINITY;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
            uint32_t r[32];
            tmem_ld32(ts + c * 32, r);
            tmem_ld_wait();
            mask_scores(r, c < 2 ? (c ? mask[1] : mask[0]) : (c == 3 ? mask[3] : mask[2]));
#pragma unroll
            for (int k = 0; k < 32; k += 2) mt = max3(mt, __uint_as_float(r[k]), __uint_as_float(r[k + 1]));
        }
        mt *= scale_log2;                                  // scale > 0
        const bool raise = row_ok && mt > m_used + kRaiseAbove;
        if (__any_sync(0xffffffffu, raise) && j > 0) {     // (nothing has been accumulated before tile 0)
            if (!mbar_wait(&sh.v_empty[(j - 1) % kWStages], (uint32_t)((j - 1) / kWStages) & 1u, sh.abort_flag, plan.wait_cycles)) return false;
            tc_fence_after_sync();
            const float alpha = raise ? exp2f(m_used - mt) : 1.f;
#pragma unroll 1
            for (int cc = 0; cc < 4; ++cc) {
                uint32_t o[32];
                tmem_ld32(tmem_o + lane_field + cc * 32, o);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                tmem_st32(tmem_o + lane_field + cc * 32, o);
            }
            tmem_st_wait();
            l *= alpha;
        }
        if (raise) m_used = mt;
        *my_ref = m_used;
        neg_m2 = pack_f32x2(-m_used, -m_used);
        uint64_t ps[2] = {0ull, 0ull};
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {                      // P of a quarter lands on scores that have been read
            uint32_t r[32], pk[16];
            tmem_ld32(ts + c * 32, r);
            tmem_ld_wait();
            mask_scores(r, c < 2 ? (c ? mask[1] : mask[0]) : (c == 3 ? mask[3] : mask[2]));
            exp_pack(r, scale2, neg_m2, pk, ps);
            tmem_st16(ts + c * 16, pk);
            tmem_st_wait();
        }
        l += sum_f32x2(add_f32x2(ps[0], ps[1]));
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0 && !(plan.withhold && j == 0)) { mbar_arrive(&sh.p_full[s]); mbar_arrive(&sh.commit[quad]); }
    }
    return true;
}

}  // namespace sdv
