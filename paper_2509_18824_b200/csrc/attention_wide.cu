// Tree-masked GQA attention with 128-key tiles: one CTA per SM, all of the SM's tensor memory.
//
// Same problem, same descriptors and same split of the work as the kernel in attention.cu (CTA = (layer,
// sequence, KV head, row tile, key chunk), chunks of a row tile form a cluster); what differs is the
// inside of a CTA.  A key tile is two 64-token cache blocks (or the last block and the tree's own keys):
// S = Q.K^T runs as eight N = 128 MMAs (64 cycles each for twice the keys an N = 64 one takes 48 for: the
// A operand is re-read from shared memory half as often), and every per-tile cost - barrier waits,
// commits, the softmax warps' waits, loads, votes and stores - is paid once per 128 keys.  Two groups of
// four softmax warps take the tiles in turn, so that one group's latencies hide behind the other's
// exponentials; three score buffers keep the tensor pipe fed while they do.  Both groups accumulate into
// the one O, which works because a row's reference stays at the first tile's maximum (see kSumLimit): the
// rare tile that raises it is serialised through a per-warp commit barrier that every tile passes anyway.
#include <atomic>
#include "attention_shared.cuh"

namespace sdv {

constexpr int kWTile = 128;                     // keys per tile: two cache blocks
constexpr int kWThreads = 289;                  // warps 0-3, 4-7 softmax groups, warp 8 TMA, warp 9 = ONE thread: MMA issuer
constexpr int kWTmaWarp = 8, kWMmaWarp = 9;
constexpr int kWStages = 3;                     // K and V ring slots, score buffers
constexpr int kWHalf = kWTile * 128;            // bytes of one D-half of a tile: [128 keys][64] bf16, swizzled (16 KiB)
constexpr int kWStage = 2 * kWHalf;             // 32 KiB
constexpr int kWQBytes = 2 * kRowTile * 128;    // 32 KiB
constexpr int kWBars = 256;                     // barriers and two words
constexpr int kWSmem = kWQBytes + 2 * kWStages * kWStage + kWBars + 3 * kRowTile * 4;   // + references, two groups' sums

template <int NL>
__global__ void __launch_bounds__(kWThreads, 1)
attn_wide_kernel(const __grid_constant__ AttnLayers<NL> layers, const sd_batch bt,
                 const float scale_log2, const AttnPlan plan, int32_t* status) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* q_smem = smem;
    uint8_t* k_smem = smem + kWQBytes;
    uint8_t* v_smem = k_smem + kWStages * kWStage;
    uint64_t* bars = reinterpret_cast<uint64_t*>(v_smem + kWStages * kWStage);
    uint64_t* k_full = bars;             // [3] TMA -> MMA
    uint64_t* v_full = bars + 3;         // [3] TMA -> MMA (and whoever clears V rows)
    uint64_t* s_full = bars + 6;         // [3] MMA -> softmax, TMA: scores of tile j in buffer j % 3, K slot j % 3 read
    uint64_t* v_empty = bars + 9;        // [3] MMA -> TMA: O updated by tile j, V slot j % 3 read
    uint64_t* p_full = bars + 12;        // [3] softmax -> MMA: P of tile j written over its scores
    uint64_t* commit = bars + 15;        // [4] per TMEM quadrant: tile j's softmax is final (phase j)
    uint64_t* o_full = bars + 19;        // MMA -> softmax (single use)
    uint64_t* q_full = bars + 20;        // TMA -> MMA
    uint64_t* x_full = bars + 21;        // clustered launches: the other chunks' rows have arrived
    uint64_t* ref_full = bars + 22;      // [4] per TMEM quadrant: the first tile's reference is known (single use)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 26);
    int* abort_flag = reinterpret_cast<int*>(bars + 27);
    int& s_seq = *reinterpret_cast<int*>(bars + 28);
    float* ref_smem = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kWBars);   // [128] by TMEM lane
    float* sum_smem = ref_smem + kRowTile;                                                   // [2][128]

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int chunk = blockIdx.x;
    const int rt = blockIdx.y;
    const int zz = (int)blockIdx.z + plan.z0;              // (sequence rank, layer, KV head), see sequence_of_rank
    const int kvh = zz % bt.Hkv;
    const int lb = zz / bt.Hkv;
    const int rank_b = lb / plan.n_layers;
    const AttnLayer& ly = layers.l[lb % plan.n_layers];

    griddep_launch_dependents();
    const bool aligned = (smem_u32(smem) & 1023u) == 0;    // swizzled tiles need 1 KiB alignment
    if (aligned) {
        if (warp == kWTmaWarp) {
            if (lane == 0) {
                *abort_flag = 0;
                for (int i = 0; i < kWStages; ++i) {
                    mbar_init(&k_full[i], 1); mbar_init(&v_full[i], 1); mbar_init(&s_full[i], 1);
                    mbar_init(&v_empty[i], 1); mbar_init(&p_full[i], 4);
                }
                for (int i = 0; i < 4; ++i) { mbar_init(&commit[i], 1); mbar_init(&ref_full[i], 1); }
                mbar_init(o_full, 1); mbar_init(q_full, 1); mbar_init(x_full, 1);
                fence_barrier_init();
                fence_proxy_async_smem();
                prefetch_tensormap(&ly.q); prefetch_tensormap(&ly.k_cache); prefetch_tensormap(&ly.v_cache);
                prefetch_tensormap(&ly.k_tree); prefetch_tensormap(&ly.v_tree);
            }
            __syncwarp();
            tmem_alloc(tmem_slot, 512);
            tmem_relinquish();
        }
    } else if (threadIdx.x == 0) {
        set_status(status, SD_ERR_UNSUPPORTED);
    }
    tc_fence_before_sync();
    __syncthreads();                                       // barriers and tensor memory are set up
    tc_fence_after_sync();
    const uint32_t tmem_base = aligned ? *tmem_slot : 0;
    const uint32_t tmem_o = tmem_base, tmem_s = tmem_base + 128;   // O, then three score buffers of 128 columns
    // A guess at the sequence's length, read while the kernel ahead may still change it: only used to fetch
    // the block table together with the real length instead of after it.
    const int len_guess = plan.ranked ? 0 : max(__ldcg(bt.len + rank_b), 0);
    griddep_wait();                                        // global memory from here on

    int b = rank_b;
    if (plan.ranked) b = sequence_of_rank(bt, rank_b, s_seq);
    const int G = bt.Hq / bt.Hkv;
    const int T = bt.T_max;
    const int tile_rows = plan.tile_rows;
    const uint64_t pol = policy_evict_first();
    if (aligned && warp == kWTmaWarp && lane == 0) {       // depends on nothing but b
        mbar_arrive_expect_tx(q_full, (uint32_t)tile_rows * kD * 2);
        tma_load_3d(q_smem, &ly.q, 0, kvh * G, b * T + rt * plan.tile_nodes, q_full, pol);
        tma_load_3d(q_smem + kRowTile * 128, &ly.q, 64, kvh * G, b * T + rt * plan.tile_nodes, q_full, pol);
    }
    const int32_t *n_nodes = bt.n_nodes, *lens = bt.len, *tables = bt.block_table;
    settle(n_nodes); settle(lens); settle(tables);         // (no load of theirs in front of the wait)
    const int n = min(max(__ldg(n_nodes + b), 0), T);
    const int len = max(__ldg(lens + b), 0);
    const int t0_guess = chunk_range(len_guess, bt.max_blocks_per_seq, chunks_of(min((len_guess + kBlock - 1) / kBlock, bt.max_blocks_per_seq), plan.n_chunks, plan.chunk_blocks), chunk).t0;
    const int32_t* const seq_table = tables + (size_t)b * bt.max_blocks_per_seq;
    int even = 0, odd = 0;                                 // block table of this chunk (producer warp)
    if (warp == kWTmaWarp) {
        if (t0_guess + lane < bt.max_blocks_per_seq) even = __ldg(seq_table + t0_guess + lane);
        if (t0_guess + 32 + lane < bt.max_blocks_per_seq) odd = __ldg(seq_table + t0_guess + 32 + lane);
    }
    const int rows = n * G;                                // rows of this sequence's own nodes
    const bool m64 = (rows - rt * tile_rows) <= 64;        // last row tile of at most 64 rows: M = 64 (lanes 0..15 of a quadrant)
    if ((len + kBlock - 1) / kBlock > bt.max_blocks_per_seq && threadIdx.x == 0) set_status(status, SD_ERR_BOUNDS);
    // key chunks of this sequence; CTAs beyond have nothing to do
    const int n_chunks = chunks_of(min((len + kBlock - 1) / kBlock, bt.max_blocks_per_seq), plan.n_chunks, plan.chunk_blocks);
    const ChunkRange cr = chunk_range(len, bt.max_blocks_per_seq, n_chunks, chunk);
    const int n_pref = cr.t1 - cr.t0;                      // cache blocks of this chunk ...
    const int nb = n_pref + (chunk == n_chunks - 1 ? 1 : 0);           // ... and the tree's keys as one more
    const int nt = (nb + 1) / 2;
    const bool has_rows = rt * tile_rows < rows && chunk < n_chunks;
    const bool active = (nt > 0) && aligned && has_rows;
    const bool clustered = (n_chunks > 1) && has_rows;     // (a CTA without work leaves; cluster barriers do not wait for it)
    const int32_t* table = seq_table + cr.t0;
    // The producer is a whole warp in uniform control flow with one lane elected around the copies (32 cycles
    // per copy; 70 from a lane-0 branch, where every operand has to be moved to uniform registers under
    // divergence, and eight copies a tile made the producer the kernel's bound).  Its lanes hold the
    // block table: 32 entries in `even` (blocks 64 w ..) and 32 in `odd` (blocks 64 w + 32 ..), fetched a
    // window ahead, handed out by shuffles.
    int jk = 0, jv = 0;
    auto window = [&](int i0) { return i0 + lane < n_pref ? __ldg(table + i0 + lane) : 0; };
    auto block_of = [&](int i) {
        int blk = __shfl_sync(0xffffffffu, (i & 32) ? odd : even, i & 31);
        if (blk < 0 || blk >= ly.num_blocks) { if (lane == 0) set_status(status, SD_ERR_BOUNDS); blk = 0; }
        return blk;
    };
    // tile j of K or V: up to two 64-key blocks into ring slot s = j % 3
    auto issue = [&](int j, int s, bool is_v) {
        const bool two = 2 * j + 1 < nb;
        uint64_t* full = (is_v ? v_full : k_full) + s;
        uint8_t* dst = (is_v ? v_smem : k_smem) + s * kWStage;
        const CUtensorMap* m = is_v ? &ly.v_cache : &ly.k_cache;
        if (2 * j + 1 < n_pref) {
            const int y0 = (block_of(2 * j) * bt.Hkv + kvh) * kBlock, y1 = (block_of(2 * j + 1) * bt.Hkv + kvh) * kBlock;
            if (elect_one()) {
                mbar_arrive_expect_tx(full, kWStage);
                tma_load_2d(dst, m, 0, y0, full, pol);
                tma_load_2d(dst + kWHalf, m, 64, y0, full, pol);
                tma_load_2d(dst + kWHalf / 2, m, 0, y1, full, pol);
                tma_load_2d(dst + kWHalf + kWHalf / 2, m, 64, y1, full, pol);
            }
        } else {                                           // the chunk's last tile: an odd block and/or the tree's keys
            const bool has0 = 2 * j < n_pref;
            const int y0 = has0 ? (block_of(2 * j) * bt.Hkv + kvh) * kBlock : 0;
            const CUtensorMap* mt = is_v ? &ly.v_tree : &ly.k_tree;
            if (elect_one()) {
                mbar_arrive_expect_tx(full, two ? kWStage : kWStage / 2);
                if (has0) {
                    tma_load_2d(dst, m, 0, y0, full, pol);
                    tma_load_2d(dst + kWHalf, m, 64, y0, full, pol);
                }
                if (!has0 || two) {
                    uint8_t* d = dst + (has0 ? kWHalf / 2 : 0);
                    tma_load_3d(d, mt, 0, kvh, b * T, full, pol);
                    tma_load_3d(d + kWHalf, mt, 64, kvh, b * T, full, pol);
                }
            }
        }
        __syncwarp();
    };
    if (chunk == 0) zero_unused_rows(bt, plan, ly, b, rt, kvh, rows, (int)threadIdx.x, kWThreads);
    float m_used = -INFINITY, l = 0.f;                     // this thread's row: reference, sum over its group's tiles
    bool rows_ready = false;

    if (active) {
    if (warp == kWTmaWarp) {
        // ------------------------------------------------------------ TMA producer
        if (cr.t0 != t0_guess) {
            even = window(0);
            odd = window(32);
        }
#pragma unroll
        for (int i = 0; i < kWStages; ++i)
            if (i < nt) {
                issue(i, i, false);
                issue(i, i, true);
                jk = jv = i + 1;
            }
        // (K slot j % 3 is free once the scores of tile j - 3 are complete: the score barrier tells both)
        bool ok = true;
        long long t_last = clock64();
        int sk = 0, sv = 0;                                // ring slots and phases of the next K and V tile
        uint32_t pk = 0, pv = 0;
        while ((jk < nt || jv < nt) && ok) {
            bool progress = false;
            if (jk < nt && __any_sync(0xffffffffu, mbar_test_wait(&s_full[sk], pk))) {
                issue(jk++, sk, false);
                if (++sk == kWStages) { sk = 0; pk ^= 1u; }
                progress = true;
            }
            if (jv < nt && __any_sync(0xffffffffu, mbar_test_wait(&v_empty[sv], pv))) {
                issue(jv, sv, true);
                // V follows K by at most three tiles: the window behind the one V has just left can be replaced
                if ((jv & 15) == 0) { if (jv & 16) even = window(2 * jv + 32); else odd = window(2 * jv + 32); }
                ++jv;
                if (++sv == kWStages) { sv = 0; pv ^= 1u; }
                progress = true;
            }
            if (progress) {
                t_last = clock64();
            } else if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(abort_flag) || clock64() - t_last > plan.wait_cycles)) {
                if (lane == 0) *reinterpret_cast<volatile int*>(abort_flag) = 1;
                ok = false;
            }
        }
        if (!ok) {
            if (lane == 0) set_status(status, SD_ERR_TIMEOUT);
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);      // let copies in flight land
        }
    } else if (warp == kWMmaWarp) {
        // ------------------------------------------------------------ MMA issuer (this warp is one thread)
        const int M = m64 ? 64 : kRowTile;
        const uint32_t idesc_s = make_idesc_bf16(M, kWTile, false, false), idesc_s_half = make_idesc_bf16(M, kWTile / 2, false, false);
        const uint32_t idesc_o = make_idesc_bf16(M, kD, false, true);
        const uint64_t qdesc = make_smem_desc(smem_u32(q_smem), 16, 1024, 128);
        const uint64_t kdesc0 = make_smem_desc(smem_u32(k_smem), 16, 1024, 128);
        const uint64_t vdesc0 = make_smem_desc(smem_u32(v_smem), kWHalf, 1024, 128);   // [key][d]: N (= d) contiguous
        bool ok = mbar_wait(q_full, 0, abort_flag, plan.wait_cycles);
        auto issue_s = [&](int j) -> bool {
            const int s = j % kWStages;
            if (!mbar_wait(&k_full[s], (uint32_t)(j / kWStages) & 1u, abort_flag, plan.wait_cycles)) return false;
            tc_fence_after_sync();
            const uint64_t kd = kdesc0 + (uint64_t)(s * (kWStage >> 4));
            const uint32_t d = tmem_s + s * kWTile;
            const uint32_t idesc = 2 * j + 1 < nb ? idesc_s : idesc_s_half;
#pragma unroll
            for (int k = 0; k < kD / 16; ++k)
                mma_ss(d, qdesc + (uint64_t)((k >> 2) * ((kRowTile * 128) >> 4) + (k & 3) * 2),
                       kd + (uint64_t)((k >> 2) * (kWHalf >> 4) + (k & 3) * 2), idesc, k != 0 ? 1u : 0u);
            mma_commit(&s_full[s]);
            return true;
        };
        for (int j = 0; j < kWStages - 1 && j < nt && ok; ++j) ok = issue_s(j);
        for (int j = 0; j < nt && ok; ++j) {
            // scores two tiles ahead: their buffer held P of tile j - 1, whose P.V was issued before
            if (j + kWStages - 1 < nt) ok = issue_s(j + kWStages - 1);
            if (!ok) break;
            const int s = j % kWStages;
            const uint32_t ph = (uint32_t)(j / kWStages) & 1u;
            if (!mbar_wait(&p_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
            if (!mbar_wait(&v_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
            tc_fence_after_sync();
            const uint64_t vd = vdesc0 + (uint64_t)(s * (kWStage >> 4));
            const uint32_t pa = tmem_s + s * kWTile;       // P from tensor memory: 16 keys = 8 columns
            const uint32_t first = (j != 0) ? 1u : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                mma_ts(tmem_o, pa + k * 8, vd + (uint64_t)(k * (2048 >> 4)), idesc_o, k != 0 ? 1u : first);
            if (2 * j + 1 < nb) {
#pragma unroll
                for (int k = 4; k < 8; ++k) mma_ts(tmem_o, pa + k * 8, vd + (uint64_t)(k * (2048 >> 4)), idesc_o, 1u);
            }
            mma_commit(&v_empty[s]);
        }
        mma_commit(o_full);
        if (!ok) {
            // unwinding: nothing may give tensor memory back while an MMA issued above still runs
            set_status(status, SD_ERR_TIMEOUT);
            mbar_wait_plain(o_full, 0, plan.wait_cycles);
        }
    } else {
        // ------------------------------------------------------------ softmax: one thread per row and group
        const int group = warp >> 2, quad = warp & 3;
        const int gt = quad * 32 + lane;                   // TMEM lane, also the index within the group
        const int row_in_tile = m64 ? (lane < 16 ? quad * 16 + lane : -1) : gt;    // -1: a TMEM lane without a row
        const int row = (row_in_tile >= 0 && row_in_tile < tile_rows) ? rt * tile_rows + row_in_tile : rows;
        const bool row_ok = row < rows;
        const uint64_t amask = row_ok ? bt.anc_mask[(size_t)b * T + plan.node_of(row)] : ~0ull;
        const uint32_t lane_field = (uint32_t)(quad * 32) << 16;
        const uint64_t scale2 = pack_f32x2(scale_log2, scale_log2);
        uint64_t neg_m2 = 0ull;                            // -(reference of this row), twice
        volatile float* my_ref = ref_smem + gt;
        bool ok = true;
        const int n_full = max(min(len / kBlock - cr.t0, n_pref), 0) / 2;   // leading tiles with all 128 keys inside the prefix
        for (int j = group; j < nt && ok; j += 2) {
            const int s = j % kWStages;
            const uint32_t ph = (uint32_t)(j / kWStages) & 1u;
            const uint32_t ts = tmem_s + lane_field + s * kWTile;
            if (j == 1) {                                  // the reference that the other group found in tile 0
                if (!mbar_wait(&ref_full[quad], 0, abort_flag, plan.wait_cycles)) { ok = false; break; }
                m_used = *my_ref;
                neg_m2 = pack_f32x2(-m_used, -m_used);
            }
            // The usual tile: all keys visible, reference known.  (See exp_pack and kSumLimit: nothing
            // but loads, exponentials and stores; masks, a new reference and clearing V rows are below.)
            if (j < n_full) {
                if (!mbar_wait(&s_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
                tc_fence_after_sync();
                if (j == 0) {                              // its maximum becomes the reference
                    float mt = -INFINITY;
#pragma unroll 1
                    for (int c = 0; c < kWTile; c += 64) {
                        uint32_t a[32], d[32];
                        tmem_ld32(ts + c, a);
                        tmem_ld32(ts + c + 32, d);
                        tmem_ld_wait();
                        float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
                        for (int k = 0; k < 32; k += 4) {
                            m0 = max3(m0, __uint_as_float(a[k]), __uint_as_float(a[k + 1]));
                            m1 = max3(m1, __uint_as_float(a[k + 2]), __uint_as_float(a[k + 3]));
                            m2 = max3(m2, __uint_as_float(d[k]), __uint_as_float(d[k + 1]));
                            m3 = max3(m3, __uint_as_float(d[k + 2]), __uint_as_float(d[k + 3]));
                        }
                        mt = max3(mt, fmaxf(m0, m1), fmaxf(m2, m3));
                    }
                    m_used = row_ok ? mt * scale_log2 : 0.f;       // scale > 0; finite for rows that nobody reads
                    *my_ref = m_used;
                    neg_m2 = pack_f32x2(-m_used, -m_used);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ref_full[quad]);   // (the other group need not wait for the tile)
                }
                uint32_t ra[16], rb[16], pk0[32], pk1[32];
                uint64_t ps[2] = {0ull, 0ull};
                tmem_ld16(ts, ra);                         // sixteen scores at a time, the next ones on their way
#pragma unroll
                for (int c = 0; c < 8; c += 2) {           // (thirty-two at a time left too few registers: spills)
                    uint32_t* pk = (c < 4 ? pk0 : pk1) + (c & 2) * 8;
                    tmem_ld_wait();
                    tmem_ld16(ts + (c + 1) * 16, rb);
                    exp_pack(ra, scale2, neg_m2, pk, ps);
                    tmem_ld_wait();
                    if (c < 6) tmem_ld16(ts + (c + 2) * 16, ra);
                    exp_pack(rb, scale2, neg_m2, pk + 8, ps);
                }
                const float psum = sum_f32x2(add_f32x2(ps[0], ps[1]));
                // the tile before is final, and its reference still the one used here
                if (j > 0 && !mbar_wait(&commit[quad], (uint32_t)(j - 1) & 1u, abort_flag, plan.wait_cycles)) { ok = false; break; }
                const float ref = *my_ref;
                if (!__any_sync(0xffffffffu, row_ok && (!(psum <= kSumLimit) || ref != m_used))) {
                    l += psum;
                    tmem_st32(ts, pk0);                    // P over the scores this thread has just consumed
                    tmem_st32(ts + 32, pk1);
                    tmem_st_wait();
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0 && !(plan.withhold && j == 0)) { mbar_arrive(&p_full[s]); mbar_arrive(&commit[quad]); }
                    continue;
                }
            }
            // Any tile.  First the V rows of keys that no row may see (cache slots at and beyond len, rows of
            // unused tree nodes): they carry weight 0, but 0 x NaN or 0 x Inf would still poison the
            // accumulator, so they are cleared in shared memory before P.V reads them (the arrival on p_full
            // orders the two).  This comes after the wait for the scores of tile j: they were issued behind
            // P.V of tile j - 3, which read the V tile that used this ring slot before, so the slot's
            // barrier is by now in the phase of tile j.
            if (!mbar_wait(&s_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
            tc_fence_after_sync();
            uint32_t mask[4];                              // visible keys of the four 32-key quarters
            int v_rows[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = 2 * j + h;
                const bool tree = i >= n_pref;
                const int valid = i >= nb ? 0 : (tree ? kBlock : max(min(len - (cr.t0 + i) * kBlock, kBlock), 0));
                v_rows[h] = i >= nb ? kBlock : (tree ? n : valid);
                const uint64_t m = (tree && i < nb) ? amask : (valid >= 64 ? ~0ull : ((1ull << valid) - 1ull));
                mask[2 * h] = (uint32_t)m; mask[2 * h + 1] = (uint32_t)(m >> 32);
            }
            if (v_rows[0] < kBlock || v_rows[1] < kBlock) {
                if (!mbar_wait(&v_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
                const int h = gt >> 6, key = gt & 63;
                if (key >= v_rows[h]) {
                    uint4* z = reinterpret_cast<uint4*>(v_smem + s * kWStage + gt * 128);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        z[c] = make_uint4(0, 0, 0, 0);
                        z[c + kWHalf / 16] = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();
                }
            }
            if (j > 0) {
                if (!mbar_wait(&commit[quad], (uint32_t)(j - 1) & 1u, abort_flag, plan.wait_cycles)) { ok = false; break; }
                const float ref = *my_ref;                 // raised by the other group since?
                if (ref != m_used) { l *= exp2f(m_used - ref); m_used = ref; }
            }
            const int n_quarters = 2 * j + 1 < nb ? 4 : 2;
            float mt = -INFINITY;
#pragma unroll 1
            for (int c = 0; c < n_quarters; ++c) {
                uint32_t r[32];
                tmem_ld32(ts + c * 32, r);
                tmem_ld_wait();
                mask_scores(r, c < 2 ? (c ? mask[1] : mask[0]) : (c == 3 ? mask[3] : mask[2]));
#pragma unroll
                for (int k = 0; k < 32; k += 2) mt = max3(mt, __uint_as_float(r[k]), __uint_as_float(r[k + 1]));
            }
            mt *= scale_log2;                              // scale > 0
            // first tile: its maximum becomes the reference; later: only a score far above it changes it
            const bool raise = row_ok && (m_used == -INFINITY || mt > m_used + kRaiseAbove) && mt > m_used;
            if (__any_sync(0xffffffffu, raise) && j > 0) {
                if (!mbar_wait(&v_empty[(j - 1) % kWStages], (uint32_t)((j - 1) / kWStages) & 1u, abort_flag, plan.wait_cycles)) { ok = false; break; }
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
            if (!row_ok) m_used = 0.f;                     // (finite exponentials for rows that nobody reads)
            *my_ref = m_used;
            neg_m2 = pack_f32x2(-m_used, -m_used);
            if (j == 0 && n_full == 0) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&ref_full[quad]);
            }
            uint64_t ps[2] = {0ull, 0ull};
#pragma unroll 1
            for (int c = 0; c < n_quarters; ++c) {         // P of a quarter lands on scores that have been read
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
            if (lane == 0 && !(plan.withhold && j == 0)) { mbar_arrive(&p_full[s]); mbar_arrive(&commit[quad]); }
        }
        // ------------------------------------------------------------ epilogue
        if (ok) ok = mbar_wait(o_full, 0, abort_flag, plan.wait_cycles);
        if (ok) {
            const float ref = *my_ref;                     // the final reference; l may still refer to an earlier one
            if (ref != m_used) { l *= exp2f(m_used - ref); m_used = ref; }
            sum_smem[group * kRowTile + gt] = l;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        ok = ok && *reinterpret_cast<volatile int*>(abort_flag) == 0;   // (uniform from here on: every failed wait raises the flag)
        if (ok) {
            l = sum_smem[gt] + sum_smem[kRowTile + gt];    // both groups' tiles, in this order
            tc_fence_after_sync();
            rows_ready = true;
            if (!clustered) {
                // Single chunk: normalise to bf16, through shared memory (the K ring is idle) so that the stores
                // to global memory are whole rows: written row by row from the threads that hold them
                // (32 rows, 16 bytes each per store) this took 4500 cycles of a CTA's 29000 at 1000 tokens.
                const int node = plan.node_of(row);
                const size_t orow = ((size_t)b * T + node) * bt.Hq + kvh * G + (row - node * G);
                const float inv = 1.f / l;
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                    uint32_t o[32];
                    tmem_ld32(tmem_o + lane_field + group * 64 + cc * 32, o);
                    tmem_ld_wait();
                    if (row_ok) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            uint32_t w[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(o[8 * c + 2 * k]) * inv,
                                                                                __uint_as_float(o[8 * c + 2 * k + 1]) * inv);
                                w[k] = *reinterpret_cast<const uint32_t*>(&hh);
                            }
                            const int piece = group * 8 + cc * 4 + c;           // 16-byte piece of the row
                            st_smem_v4(smem_u32(k_smem) + row_in_tile * 256 + ((piece ^ (row_in_tile & 7)) << 4), w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
                const int out_rows = min(rows - rt * tile_rows, tile_rows);
                for (int i = (int)threadIdx.x; i < out_rows * 16; i += 256) {
                    const int r = i >> 4, piece = i & 15, rr = rt * tile_rows + r, nd = plan.node_of(rr);
                    const size_t at = ((size_t)b * T + nd) * bt.Hq + kvh * G + (rr - nd * G);
                    reinterpret_cast<float4*>(ly.out + at * kD)[piece] = ld_smem_v4(smem_u32(k_smem) + r * 256 + ((piece ^ (r & 7)) << 4));
                }
                if (row_ok && ly.lse && group == 0) ly.lse[orow] = (m_used + log2f(l)) * 0.6931471805599453f;
            }
        } else if (lane == 0) {
            set_status(status, SD_ERR_TIMEOUT);
        }
    }
    }   // active

    if (!active && aligned && warp == kWTmaWarp && lane == 0)      // nobody else waits for the Q copy
        mbar_wait(q_full, 0, abort_flag, plan.wait_cycles);

    if (clustered) {
        // The chunks' rows meet as described at exchange_rows; the rings are free by now.
        const int gt = (int)threadIdx.x & 127;
        const int row_in_tile = m64 ? (lane < 16 ? (warp & 3) * 16 + lane : -1) : gt;
        const RowExchange x{bt, plan, ly, smem_u32(k_smem), smem_u32(x_full), chunk, n_chunks, rt, b, kvh, rows, cr.tpc, cr.tiles_total};
        if (threadIdx.x == 0) exchange_expect(x, x_full);
        __syncwarp();
        cluster_arrive_release();                          // every CTA's MMAs and copies are complete
        cluster_wait_acquire();
        if (active && warp < 8)
            exchange_push<2>(x, tmem_base + ((uint32_t)((warp & 3) * 32) << 16), (warp >> 2) * 2, rows_ready, row_in_tile, m_used, l);
        __syncwarp();
        cluster_arrive_relaxed();                          // (waited for at the end: nobody leaves before its peers have sent)
        if (warp < 8) {
            asm volatile("bar.sync 1, 256;" ::: "memory"); // this CTA's own rows
            if (mbar_wait_cluster(x_full, 0, abort_flag, plan.wait_cycles)) {
                if (n_chunks == 2) merge_rows<2, 256>(x, (int)threadIdx.x);
                else if (n_chunks == 4) merge_rows<4, 256>(x, (int)threadIdx.x);
                else merge_rows<8, 256>(x, (int)threadIdx.x);
            } else if (lane == 0) {
                set_status(status, SD_ERR_TIMEOUT);
                for (int i = 0; i < 1000; ++i) __nanosleep(1000);      // let rows in flight land
            }
        }
        __syncwarp();
        cluster_wait_acquire();
    }
    if (!aligned) return;
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kWTmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

template <int NL>
sd_status launch_wide(const AttnLayers<NL>& layers, const sd_batch& bt, float scale, const AttnPlan& plan,
                      int z_count, int32_t* dev_status, cudaStream_t st) {
    return launch_attn(attn_wide_kernel<NL>, kWThreads, kWSmem, layers, bt, scale, plan, z_count, dev_status, st);
}
template sd_status launch_wide<1>(const AttnLayers<1>&, const sd_batch&, float, const AttnPlan&, int, int32_t*, cudaStream_t);
template sd_status launch_wide<kMaxLayersPerLaunch>(const AttnLayers<kMaxLayersPerLaunch>&, const sd_batch&, float,
                                                    const AttnPlan&, int, int32_t*, cudaStream_t);

// Clusters of n_chunks CTAs that the current device runs at a time (asked once per device and size: with one
// CTA per SM it depends on how many SMs each GPC has; 8 x 16 of the 148 do not all fit, for instance).
int wide_resident_clusters(int dev, int sms, int n_chunks) {
    constexpr int kDevs = 64;
    static std::atomic<int> cache[kDevs][4];
    if (n_chunks <= 1) return sms;
    const int slot = n_chunks == 2 ? 1 : (n_chunks == 4 ? 2 : 3);
    if (dev >= 0 && dev < kDevs)
        if (const int v = cache[dev][slot].load(std::memory_order_relaxed)) return v;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_chunks, 1, sms);
    cfg.blockDim = dim3(kWThreads);
    cfg.dynamicSmemBytes = kWSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = n_chunks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(attn_wide_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, attn_wide_kernel<1>, &cfg) != cudaSuccess || n < 1)
        n = max(1, sms / n_chunks - n_chunks);             // (no answer: a cautious guess, and ask again next time)
    else if (dev >= 0 && dev < kDevs)
        cache[dev][slot].store(n, std::memory_order_relaxed);
    return n;
}

}  // namespace sdv
