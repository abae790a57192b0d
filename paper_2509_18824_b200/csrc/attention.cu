// Tree-masked GQA attention over a paged prefix cache plus the tree's own KV,
// on the 5th-generation tensor cores (tcgen05 + TMEM), split-KV.
//
// All T*G query rows that share one KV head (node-major: row = node*G + g) are
// processed against every K/V byte exactly once per 128-row tile: with 60 nodes
// and 7 grouped heads that is 420 rows per K/V row, which makes the step
// compute-bound, so both S = Q.K^T and O += P.V run as tcgen05.mma with
// accumulators in TMEM.
//
// One CTA = (sequence, KV head, 128-row tile, key chunk).  Its key tiles are the
// 64-token cache blocks of the chunk (TMA, 128-byte swizzle, located through the
// block table) and, for the last chunk, one extra tile holding the tree's own
// keys, masked per row by the node's ancestor bitmask.  Softmax runs one thread
// per row straight out of TMEM (no cross-thread reductions); the row's reference is
// the maximum of its first tile and is raised only when a tile's sum leaves the
// safe range, so the accumulator in TMEM is practically never rescaled.  P goes back into TMEM and feeds the second MMA from there.
// With one chunk the CTA writes the output itself; otherwise the chunks of a row
// tile form a thread-block cluster: every CTA pushes its (max, sum, unnormalised
// O) rows into the shared memory of the CTA that finishes them (remote stores),
// and each CTA merges its share of the rows locally, in chunk order.
// The launch is a programmatic dependent launch: barriers, tensor memory and
// tensor-map prefetch are set up before the kernel waits for the kernel ahead of
// it in the stream, so consecutive per-layer calls overlap their ends.
#include "attention_plan.cuh"

namespace sdv {

constexpr int kKeyTile = 64;                   // keys per tile = one cache block
constexpr int kAttThreads = 161;               // warps 0-3 softmax, warp 4 TMA, warp 5 = ONE thread: MMA issuer
constexpr int kTmaWarp = 4, kMmaWarp = 5;
constexpr int kSubTile = kKeyTile * 128;       // bytes of a [64][64] bf16 swizzled sub-tile (8 KiB)
constexpr int kQBytes = 2 * kRowTile * 128;    // Q tile: two D-halves of [128][64] bf16 (32 KiB)
constexpr int kKVStage = 2 * kSubTile;         // one K (or V) tile: two D-halves (16 KiB)
constexpr int kKStages = 3;                    // K tiles are consumed a tile ahead of V
constexpr int kVStages = 2;
constexpr int kAttSmem = kQBytes + (kKStages + kVStages) * kKVStage + 256;
constexpr int kTmemCols = 256;                 // O: 0..127, S/P buffers: 128..191, 192..255
// P (bf16, two keys per 32-bit column) overwrites the first 32 columns of the S buffer it came from

template <int NL>
__global__ void __launch_bounds__(kAttThreads, 2)
attn_umma_kernel(const __grid_constant__ AttnLayers<NL> layers, const sd_batch bt,
                 const float scale_log2, const AttnPlan plan, int32_t* status) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* q_smem = smem;
    uint8_t* k_smem = smem + kQBytes;
    uint8_t* v_smem = k_smem + kKStages * kKVStage;
    uint64_t* bars = reinterpret_cast<uint64_t*>(v_smem + kVStages * kKVStage);
    uint64_t* k_full = bars;             // [3] TMA -> MMA
    uint64_t* k_empty = bars + 3;        // [3] MMA -> TMA
    uint64_t* v_full = bars + 6;         // [2]
    uint64_t* v_empty = bars + 8;        // [2]
    uint64_t* s_full = bars + 10;        // [2] MMA -> softmax (scores of tile j in buffer j&1)
    uint64_t* p_full = bars + 12;        // [2] softmax -> MMA (P written into buffer j&1, O rescaled); one
                                         //     barrier per buffer so that a warp running a tile ahead
                                         //     cannot complete the previous tile's phase
    uint64_t* pv_done = bars + 14;       // MMA -> softmax   (O updated by tile j; phase j)
    uint64_t* o_full = bars + 15;        // MMA -> softmax   (single use: every MMA of the CTA has completed)
    uint64_t* q_full = bars + 16;        // TMA -> MMA       (Q tile)
    uint64_t* x_full = bars + 20;        // clustered launches: the other chunks' rows have arrived (single use)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 17);
    int* abort_flag = reinterpret_cast<int*>(bars + 18);

    // warp index as a value the compiler knows to be warp-uniform, so that role dispatch is uniform
    // control flow (a warp's non-existent lanes do not take part in the shuffle)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const int chunk = blockIdx.x;
    const int rt = blockIdx.y;
    // blockIdx.z enumerates (sequence rank, layer, KV head), see sequence_of_rank
    const int zz = (int)blockIdx.z + plan.z0;
    const int kvh = zz % bt.Hkv;
    const int lb = zz / bt.Hkv;
    const int rank_b = lb / plan.n_layers;
    const AttnLayer& ly = layers.l[lb % plan.n_layers];
    const CUtensorMap* const map_q = &ly.q;
    const CUtensorMap* const map_kc = &ly.k_cache;
    const CUtensorMap* const map_vc = &ly.v_cache;
    const CUtensorMap* const map_kt = &ly.k_tree;
    const CUtensorMap* const map_vt = &ly.v_tree;

    // Set-up that touches no global memory comes first: when the launch is allowed to start before the
    // kernel ahead of it in the stream has finished (programmatic dependent launch: one attention call
    // per layer, back to back), it overlaps that kernel's tail.  The kernel behind this one may start
    // its own set-up as soon as every CTA of this grid is running.
    griddep_launch_dependents();
    const bool aligned = (smem_u32(smem) & 1023u) == 0;    // swizzled tiles need 1 KiB alignment
    uint32_t tmem_base = 0;
    if (aligned) {
        if (warp == kTmaWarp) {                            // a full warp (the MMA warp is a single thread)
            if (lane == 0) {                               // (this thread uses some of them before the block meets)
                *abort_flag = 0;
                for (int i = 0; i < kKStages; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1); }
                for (int i = 0; i < kVStages; ++i) { mbar_init(&v_full[i], 1); mbar_init(&v_empty[i], 1); }
                for (int i = 0; i < 2; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 4); }
                mbar_init(pv_done, 1); mbar_init(q_full, 1); mbar_init(o_full, 1); mbar_init(x_full, 1);
                fence_barrier_init();
                fence_proxy_async_smem();
                prefetch_tensormap(map_q); prefetch_tensormap(map_kc); prefetch_tensormap(map_vc);
                prefetch_tensormap(map_kt); prefetch_tensormap(map_vt);
            }
            __syncwarp();
            tmem_alloc(tmem_slot, kTmemCols);
            tmem_relinquish();
        }
    } else if (threadIdx.x == 0) {
        set_status(status, SD_ERR_UNSUPPORTED);
    }
    // everything below reads (or writes) global memory that the kernel ahead may still be working on
    griddep_wait();

    // (the slot lives in the dynamic shared-memory block: a static variable would push that block's
    //  1 KiB-aligned start and cost the second resident CTA)
    int b = rank_b;
    if (plan.ranked) b = sequence_of_rank(bt, rank_b, *reinterpret_cast<int*>(bars + 19));
    __nv_bfloat16* __restrict__ out = ly.out;
    float* __restrict__ lse = ly.lse;
    const int num_blocks = ly.num_blocks;
    const int G = bt.Hq / bt.Hkv;
    const int T = bt.T_max;
    // The Q tile depends on nothing but b, so it is requested before the lengths are known: one copy of
    // whole nodes (tile_rows = the largest multiple of G up to 128; rows of unused nodes are loaded too and
    // reach no output, the smem rows behind tile_rows hold whatever they held).  (Staged through registers
    // by the softmax threads it took two more dependent memory latencies before the first scores.)
    const int tile_rows = plan.tile_rows;
    const uint64_t pol = policy_evict_first();
    if (aligned && warp == kTmaWarp && lane == 0) {
        mbar_arrive_expect_tx(q_full, (uint32_t)tile_rows * kD * 2);
        tma_load_3d(q_smem, map_q, 0, kvh * G, b * T + rt * plan.tile_nodes, q_full, pol);
        tma_load_3d(q_smem + kRowTile * 128, map_q, 64, kvh * G, b * T + rt * plan.tile_nodes, q_full, pol);
    }
    const int32_t *n_nodes = bt.n_nodes, *lens = bt.len, *tables = bt.block_table;
    settle(n_nodes); settle(lens); settle(tables);         // (no load of theirs in front of the wait)
    // (lengths that a kernel of this library wrote while this one was already there: not for the read-only path)
    const int n = min(max(__ldcg(n_nodes + b), 0), T);
    const int len = max(__ldcg(lens + b), 0);
    // Rows of this sequence: its own nodes only (rows are node-major, so they are the first n * G).  A tree
    // smaller than T_max pays for the row tiles it fills: the rows behind them only get their zeros.  (A
    // batch of 16 trees of 30 to 60 nodes, T_max = 60: 2.9 of 4 row tiles run.)
    const int rows = n * G;
    // A last row tile of at most 64 rows (420 rows = 3 x 128 + 36) runs its MMAs with M = 64: the
    // accumulator rows then sit in lanes 0..15 of each 32-lane TMEM quadrant (row = 16 * quadrant + lane),
    // the tensor cores work at half width and only 64 rows of Q are staged and re-read per key tile.
    const bool m64 = (rows - rt * tile_rows) <= 64;

    // key tiles of this CTA: cache blocks [t0, t1) and, for the last chunk, the tree tile
    if ((len + kKeyTile - 1) / kKeyTile > bt.max_blocks_per_seq && threadIdx.x == 0)
        set_status(status, SD_ERR_BOUNDS);                 // the block table does not cover this length
    const ChunkRange cr = chunk_range(plan, len, bt.max_blocks_per_seq, chunk);
    const int n_chunks = cr.n_chunks;                      // of this sequence; CTAs beyond have nothing to do
    const int tiles_total = cr.tiles_total, tpc = cr.tpc, t0 = cr.t0, t1 = cr.t1;
    const bool has_tree = (chunk == n_chunks - 1);
    const int nt = (t1 - t0) + (has_tree ? 1 : 0);
    // A CTA without key tiles has nothing to compute, but it still takes part in the cluster barriers; a
    // row tile without rows is skipped by every CTA of its cluster.
    const bool has_rows = rt * tile_rows < rows && chunk < n_chunks;
    const bool active = (nt > 0) && aligned && has_rows;
    const bool clustered = (n_chunks > 1) && has_rows;   // cluster = the chunks of one (b, kvh, row tile)
    // The producer thread fills the rings before the block meets: K and V tiles travel through separate
    // rings and are issued independently, whichever slot frees first: the next K tile (needed early, for
    // the score MMA issued one tile ahead) must not queue behind a V slot that is only released when P.V
    // has finished.  The block table is looked up ahead of its use (the first entries all at once).
    const int32_t* table = tables + (size_t)b * bt.max_blocks_per_seq;
    const int n_pref = t1 - t0;
    int jk = 0, jv = 0, blk_k = 0, blk_v = 0;
    auto issue = [&](int j, int blk, bool is_v) {
        const int stages = is_v ? kVStages : kKStages;
        const int s = j % stages;
        uint64_t* full = (is_v ? v_full : k_full) + s;
        uint8_t* dst = (is_v ? v_smem : k_smem) + s * kKVStage;
        mbar_arrive_expect_tx(full, kKVStage);
        if (j >= n_pref) {
            const CUtensorMap* m = is_v ? map_vt : map_kt;
            tma_load_3d(dst, m, 0, kvh, b * T, full, pol);
            tma_load_3d(dst + kSubTile, m, 64, kvh, b * T, full, pol);
        } else {
            if (blk < 0 || blk >= num_blocks) { set_status(status, SD_ERR_BOUNDS); blk = 0; }
            const CUtensorMap* m = is_v ? map_vc : map_kc;
            const int y = (blk * bt.Hkv + kvh) * kKeyTile;
            tma_load_2d(dst, m, 0, y, full, pol);
            tma_load_2d(dst + kSubTile, m, 64, y, full, pol);
        }
    };
    if (active && warp == kTmaWarp && lane == 0) {
        int first[kKStages + 1];
#pragma unroll
        for (int i = 0; i <= kKStages; ++i) first[i] = i < n_pref ? __ldg(table + t0 + i) : 0;
        blk_k = kKStages < n_pref ? first[kKStages] : 0;
        blk_v = kVStages < n_pref ? first[kVStages] : 0;
#pragma unroll
        for (int i = 0; i < kKStages; ++i) {
            if (i < nt) { issue(i, first[i], false); jk = i + 1; }
            if (i < kVStages && i < nt) { issue(i, first[i], true); jv = i + 1; }
        }
    }
    if (chunk == 0) zero_unused_rows(bt, plan, ly, b, rt, kvh, rows, (int)threadIdx.x, kAttThreads);
    float m_used = -INFINITY, l = 0.f;                     // softmax state of this thread's row (warps 0-3)
    bool rows_ready = false;                               // ... and whether it completed (clustered launches)

    // the set-up at the top (barriers, tensor memory) is visible to every thread from here on
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (aligned) tmem_base = *tmem_slot;
    const uint32_t tmem_o = tmem_base;
    const uint32_t tmem_s = tmem_base + 128;

    if (active) {
    if (warp == kTmaWarp) {
        // ------------------------------------------------------------ TMA producer (one thread)
        if (lane == 0) {
            bool ok = true;
            long long t_last = clock64();
            while ((jk < nt || jv < nt) && ok) {
                bool progress = false;
                if (jk < nt && mbar_test_wait(&k_empty[jk % kKStages], ((uint32_t)(jk / kKStages) & 1u) ^ 1u)) {
                    issue(jk, blk_k, false);
                    ++jk;
                    if (jk < n_pref) blk_k = __ldg(table + t0 + jk);
                    progress = true;
                }
                if (jv < nt && mbar_test_wait(&v_empty[jv % kVStages], ((uint32_t)(jv / kVStages) & 1u) ^ 1u)) {
                    issue(jv, blk_v, true);
                    ++jv;
                    if (jv < n_pref) blk_v = __ldg(table + t0 + jv);
                    progress = true;
                }
                if (progress) {
                    t_last = clock64();
                } else if (*reinterpret_cast<volatile int*>(abort_flag) || clock64() - t_last > plan.wait_cycles) {
                    *reinterpret_cast<volatile int*>(abort_flag) = 1;
                    ok = false;
                }
            }
            if (!ok) {
                set_status(status, SD_ERR_TIMEOUT);
                unwind_pause();
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        // This warp consists of one thread (the block has 5 * 32 + 1 threads), so everything in
        // here is uniform control flow on warp-uniform values: tcgen05.mma takes its descriptors
        // from uniform registers, and inside a divergent "lane 0 only" region of a full warp every
        // descriptor would first have to be moved there, instruction by instruction.
        {
            const uint32_t idesc_s = make_idesc_bf16(m64 ? 64 : kRowTile, kKeyTile, false, false);   // S = Q . K^T
            const uint32_t idesc_o = make_idesc_bf16(m64 ? 64 : kRowTile, kD, false, true);          // O += P . V
            // k-steps only move the (16-byte granular) start-address field in the low bits
            const uint64_t qdesc_base = make_smem_desc(smem_u32(q_smem), 16, 1024, 128);
            const uint64_t kdesc_base = make_smem_desc(smem_u32(k_smem), 16, 1024, 128);
            // V is stored [key][d]: N (= d) contiguous; D-halves kSubTile apart, 8-key groups 1 KiB apart
            const uint64_t vdesc_base = make_smem_desc(smem_u32(v_smem), kSubTile, 1024, 128);
            bool ok = mbar_wait(q_full, 0, abort_flag, plan.wait_cycles);
            auto issue_s = [&](int j) -> bool {
                const int s = j & 1;                               // score buffer
                const int ks = j % kKStages;                       // K ring slot
                if (!mbar_wait(&k_full[ks], (uint32_t)(j / kKStages) & 1u, abort_flag, plan.wait_cycles)) return false;
                tc_fence_after_sync();
                const uint64_t kd = kdesc_base + (uint64_t)(ks * (kKVStage >> 4));
                const uint32_t d = tmem_s + s * kKeyTile;
#pragma unroll
                for (int k = 0; k < kD / 16; ++k)
                    mma_ss(d, qdesc_base + (uint64_t)((k >> 2) * ((kRowTile * 128) >> 4) + (k & 3) * 2),
                           kd + (uint64_t)((k >> 2) * (kSubTile >> 4) + (k & 3) * 2), idesc_s, k != 0 ? 1u : 0u);
                mma_commit(&k_empty[ks]);
                mma_commit(&s_full[s]);
                return true;
            };
            if (ok) ok = issue_s(0);
            for (int j = 0; j < nt && ok; ++j) {
                if (j + 1 < nt) ok = issue_s(j + 1);
                if (!ok) break;
                const int s = j & 1;
                const uint32_t ph = (uint32_t)(j >> 1) & 1u;
                if (!mbar_wait(&p_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
                const int vs = j % kVStages;
                if (!mbar_wait(&v_full[vs], (uint32_t)(j / kVStages) & 1u, abort_flag, plan.wait_cycles)) { ok = false; break; }
                tc_fence_after_sync();
                const uint64_t vd = vdesc_base + (uint64_t)(vs * (kKVStage >> 4));
                const uint32_t pa = tmem_s + s * kKeyTile;        // P comes straight from TMEM: 16 keys = 8 columns
                const uint32_t first = (j != 0) ? 1u : 0u;
#pragma unroll
                for (int k = 0; k < kKeyTile / 16; ++k)
                    mma_ts(tmem_o, pa + k * 8, vd + (uint64_t)(k * (2048 >> 4)), idesc_o, k != 0 ? 1u : first);
                mma_commit(&v_empty[vs]);
                mma_commit(pv_done);
            }
            mma_commit(o_full);
            if (!ok) {
                // unwinding: nothing may give tensor memory back while an MMA issued above still runs
                set_status(status, SD_ERR_TIMEOUT);
                mbar_wait_plain(o_full, 0, plan.wait_cycles);
                unwind_pause();
            }
        }
    } else if (warp < 4) {
        // ------------------------------------------------------------ softmax: one thread per row
        const int tid = warp * 32 + lane;
        const int row_in_tile = m64 ? (lane < 16 ? warp * 16 + lane : -1) : tid;   // -1: a TMEM lane without a row
        const int row = (row_in_tile >= 0 && row_in_tile < tile_rows) ? rt * tile_rows + row_in_tile : rows;
        const int node = row / G;
        const int g = row - node * G;
        const bool row_ok = row < rows;
        if (!row_ok) m_used = 0.f;                             // (finite exponentials for rows that nobody reads)
        const uint64_t amask = row_ok ? bt.anc_mask[(size_t)b * T + node] : ~0ull;
        const uint32_t lane_field = (uint32_t)(warp * 32) << 16;
        const uint64_t scale2 = pack_f32x2(scale_log2, scale_log2);
        uint64_t neg_m2 = 0ull;                                // -(reference of this row), twice
        bool ok = true;
        const int n_full = max(min(len / kKeyTile - t0, n_pref), 0);    // leading tiles whose 64 keys are all inside the prefix
        for (int j = 0; j < nt && ok; ++j) {
            const int s = j & 1;
            const uint32_t ph = (uint32_t)(j >> 1) & 1u;
            // The usual tile (all keys visible, reference known): nothing but loads, exponentials and stores.
            // Masks, a new reference and clearing V rows live in the other body below; as branches inside
            // one body they cost every tile 370 of 1600 cycles (predicated masks, scores kept alive).
            // The exponentials are taken against the row's reference straight away.  The reference is the
            // maximum of the first tile and need not follow later ones: P (bf16) and the sums (fp32) have
            // fp32's exponent range, so their relative precision does not depend on how far a score lies
            // above the reference.  Only when the tile's sum leaves the safe range (> 2^40: some score more
            // than about 34 powers of two above the reference) is the reference raised and the tile redone
            // (its scores are still in tensor memory).  The sum is needed anyway, so no maximum is tracked,
            // and scaling and sums run two elements per instruction.
            if (j > 0 && j < n_full) {
                if (!mbar_wait(&s_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
                tc_fence_after_sync();
                uint32_t r0[32], r1[32], pk[32];
                uint64_t ps[2] = {0ull, 0ull};
                tmem_ld32(tmem_s + lane_field + s * kKeyTile, r0);
                tmem_ld_wait();
                tmem_ld32(tmem_s + lane_field + s * kKeyTile + 32, r1);   // in flight while the first half is processed
                exp_pack(r0, scale2, neg_m2, pk, ps);
                tmem_ld_wait();
                exp_pack(r1, scale2, neg_m2, pk + 16, ps);
                const float psum = sum_f32x2(add_f32x2(ps[0], ps[1]));
                // (padding rows have harmless scores; NaN scores of a real row take the other body and stay NaN)
                if (!__any_sync(0xffffffffu, row_ok && !(psum <= kSumLimit))) {
                    l += psum;
                    // P replaces the S columns this thread has just consumed (its own TMEM lane)
                    tmem_st32(tmem_s + lane_field + s * kKeyTile, pk);
                    tmem_st_wait();
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&p_full[s]);
                    continue;
                }
            }
            const bool tree = (j >= t1 - t0);
            const int valid = tree ? kKeyTile : len - (t0 + j) * kKeyTile;   // keys of this block inside the prefix
            if (!mbar_wait(&s_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
            tc_fence_after_sync();
            // Keys that no row may see (cache slots at and beyond len, rows of unused tree nodes) carry
            // weight 0, but 0 x NaN or 0 x Inf would still poison the accumulator: their V rows are
            // cleared in shared memory before P.V reads them (the arrival on p_full below orders the
            // two), so those slots may hold any bit pattern.  This comes after the wait for the scores
            // of tile j: they were issued behind P.V of tile j - 2, which read the V tile that used this
            // ring slot before, so the slot's barrier is by now in the phase of tile j and the parity
            // wait below cannot be taken for an earlier phase.  A key row is 128 contiguous bytes in each
            // of the two D-halves (the swizzle stays inside a row).
            const int v_rows = tree ? n : valid;
            if (v_rows < kKeyTile && warp < 2) {                     // threads 0..63 <-> key rows
                const int vs = j % kVStages;
                if (!mbar_wait(&v_full[vs], (uint32_t)(j / kVStages) & 1u, abort_flag, plan.wait_cycles)) { ok = false; break; }
                if (tid >= v_rows) {
                    uint4* z = reinterpret_cast<uint4*>(v_smem + vs * kKVStage + tid * 128);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        z[c] = make_uint4(0, 0, 0, 0);
                        z[c + kSubTile / 16] = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();
                }
            }
            uint32_t r0[32], r1[32], pk[32];
            tmem_ld32(tmem_s + lane_field + s * kKeyTile, r0);
            tmem_ld32(tmem_s + lane_field + s * kKeyTile + 32, r1);
            tmem_ld_wait();
            if (tree || valid < kKeyTile) {
                mask_scores(r0, tree ? (uint32_t)amask : (valid >= 32 ? ~0u : ((1u << max(valid, 0)) - 1u)));
                mask_scores(r1, tree ? (uint32_t)(amask >> 32)
                                     : (valid >= 64 ? ~0u : (valid <= 32 ? 0u : ((1u << (valid - 32)) - 1u))));
            }
            uint64_t ps[2] = {0ull, 0ull};
            if (j > 0) {
                exp_pack(r0, scale2, neg_m2, pk, ps);
                exp_pack(r1, scale2, neg_m2, pk + 16, ps);
            }
            float psum = sum_f32x2(add_f32x2(ps[0], ps[1]));
            bool raise = row_ok && (j == 0 || !(psum <= kSumLimit));
            if (__any_sync(0xffffffffu, raise)) {
                float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    mx[c & 3] = max3(mx[c & 3], __uint_as_float(r0[2 * c]), __uint_as_float(r0[2 * c + 1]));
                    mx[(c + 2) & 3] = max3(mx[(c + 2) & 3], __uint_as_float(r1[2 * c]), __uint_as_float(r1[2 * c + 1]));
                }
                const float mt = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale_log2;   // scale > 0
                raise = raise && mt > m_used;
                if (j > 0) {
                    if (!mbar_wait(pv_done, (uint32_t)(j - 1) & 1u, abort_flag, plan.wait_cycles)) { ok = false; break; }
                    tc_fence_after_sync();
                    const float alpha = raise ? exp2f(m_used - mt) : 1.f;
#pragma unroll
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
                neg_m2 = pack_f32x2(-m_used, -m_used);
                // (again) against the new reference: the same values for rows that did not raise
                ps[0] = ps[1] = 0ull;
                exp_pack(r0, scale2, neg_m2, pk, ps);
                exp_pack(r1, scale2, neg_m2, pk + 16, ps);
                psum = sum_f32x2(add_f32x2(ps[0], ps[1]));
            }
            l += psum;
            // P replaces the S columns this thread has just consumed (its own TMEM lane)
            tmem_st32(tmem_s + lane_field + s * kKeyTile, pk);
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0 && !(plan.withhold && j == 0)) mbar_arrive(&p_full[s]);
        }
        // ------------------------------------------------------------ epilogue
        // (a parity wait on pv_done would be ambiguous here: the softmax may be two phases ahead of it)
        if (ok) ok = mbar_wait(o_full, 0, abort_flag, plan.wait_cycles);
        if (ok && !clustered) {
            // single chunk: normalise and write bf16 output
            tc_fence_after_sync();
            const int h = kvh * G + g;
            const size_t orow = ((size_t)b * T + node) * bt.Hq + h;
            const float inv = 1.f / l;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                uint32_t o[32];
                tmem_ld32(tmem_o + lane_field + cc * 32, o);
                tmem_ld_wait();
                if (row_ok) {
                    uint32_t w[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(o[2 * c]) * inv, __uint_as_float(o[2 * c + 1]) * inv);
                        w[c] = *reinterpret_cast<uint32_t*>(&hh);
                    }
                    uint4* dst = reinterpret_cast<uint4*>(out + orow * kD + cc * 32);
#pragma unroll
                    for (int c = 0; c < 4; ++c) dst[c] = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                }
            }
            if (row_ok && lse) lse[orow] = (m_used + log2f(l)) * 0.6931471805599453f;
        } else if (ok) {
            rows_ready = true;         // several chunks: the rows leave for their finishing CTAs below
        } else {
            if (lane == 0) set_status(status, SD_ERR_TIMEOUT);
            unwind_pause();
        }
    }
    }   // active

    if (!active && aligned && warp == kTmaWarp && lane == 0 && !mbar_wait(q_full, 0, abort_flag, plan.wait_cycles)) {   // nobody else waits for the Q copy
        set_status(status, SD_ERR_TIMEOUT);
        unwind_pause();
    }

    if (clustered) {
        // The chunks' rows meet as described at RowExchange; the rings are free by now.
        const RowExchange x{bt, plan, ly, smem_u32(k_smem), smem_u32(x_full), chunk, n_chunks, rt, b, kvh, rows, tpc, tiles_total};
        if (threadIdx.x == 0) exchange_expect(x, x_full);
        __syncwarp();
        cluster_arrive_release();                          // every CTA's MMAs and copies are complete
        cluster_wait_acquire();
        if (active && warp < 4)
            exchange_push<4>(x, tmem_base + ((uint32_t)(warp * 32) << 16), 0, rows_ready,
                             m64 ? (lane < 16 ? warp * 16 + lane : -1) : (int)threadIdx.x, m_used, l);
        __syncwarp();
        cluster_arrive_relaxed();                          // (waited for at the end: nobody leaves before its peers have sent)
        bool late = false;
        if (warp < 4) {
            asm volatile("bar.sync 1, 128;" ::: "memory"); // this CTA's own rows
            if (mbar_wait_cluster(x_full, 0, abort_flag, plan.wait_cycles)) {
                if (n_chunks == 2) merge_rows<2, 128>(x, (int)threadIdx.x);
                else if (n_chunks == 4) merge_rows<4, 128>(x, (int)threadIdx.x);
                else merge_rows<8, 128>(x, (int)threadIdx.x);
            } else if (lane == 0) {
                set_status(status, SD_ERR_TIMEOUT);
                late = true;
            }
        }
        __syncwarp();
        cluster_wait_acquire();
        if (late) unwind_pause();                          // (rows sent by now)
    }
    if (!aligned) return;
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kTmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

static bool fill_layer(AttnLayer* ly, const sd_batch& bt, const sd_kv_layer& cache, const void* q,
                       const void* kt, const void* vt, void* out, float* lse) {
    const int G = bt.Hq / bt.Hkv;
    const uint64_t q_dims[3] = {(uint64_t)kD, (uint64_t)bt.Hq, (uint64_t)bt.B * bt.T_max};
    const uint64_t q_strides[2] = {(uint64_t)kD * 2, (uint64_t)bt.Hq * kD * 2};
    const uint32_t q_box[3] = {64, (uint32_t)G, (uint32_t)(kRowTile / G)};
    if (!encode_tmap_bf16_3d(&ly->q, q, q_dims, q_strides, q_box, 128)) return false;
    const uint64_t cache_rows = (uint64_t)cache.num_blocks * bt.Hkv * kKeyTile;
    if (!encode_tmap_bf16_2d(&ly->k_cache, cache.k, cache_rows, kD, kD * 2, 64, kKeyTile, 128) ||
        !encode_tmap_bf16_2d(&ly->v_cache, cache.v, cache_rows, kD, kD * 2, 64, kKeyTile, 128))
        return false;
    const uint64_t dims[3] = {(uint64_t)kD, (uint64_t)bt.Hkv, (uint64_t)bt.B * bt.T_max};
    const uint64_t strides[2] = {(uint64_t)kD * 2, (uint64_t)bt.Hkv * kD * 2};
    const uint32_t box[3] = {64, 1, kKeyTile};
    if (!encode_tmap_bf16_3d(&ly->k_tree, kt, dims, strides, box, 128) ||
        !encode_tmap_bf16_3d(&ly->v_tree, vt, dims, strides, box, 128))
        return false;
    ly->out = static_cast<__nv_bfloat16*>(out);
    ly->lse = lse;
    ly->num_blocks = cache.num_blocks;
    return true;
}

template <int NL>
sd_status launch_rows1(const AttnLayers<NL>& layers, const sd_batch& bt, float scale, const AttnPlan& plan,
                       int z_count, int32_t* dev_status, cudaStream_t st) {
    return launch_attn(attn_umma_kernel<NL>, kAttThreads, kAttSmem, layers, bt, scale, plan, z_count, dev_status, st);
}
template sd_status launch_rows1<1>(const AttnLayers<1>&, const sd_batch&, float, const AttnPlan&, int, int32_t*,
                                   cudaStream_t);
template sd_status launch_rows1<kMaxLayersPerLaunch>(const AttnLayers<kMaxLayersPerLaunch>&, const sd_batch&, float,
                                                     const AttnPlan&, int, int32_t*, cudaStream_t);

// The chunks of a row tile are merged inside a thread-block cluster, through shared memory:
// attention needs no global scratch (a nominal size keeps the argument checks uniform).
size_t attention_workspace_bytes(const sd_batch&) { return 256; }

static AttnPlan common_plan(const sd_batch& bt, int n_layers, const TestKnobs& knobs) {
    AttnPlan p;
    const int G = bt.Hq / bt.Hkv;
    p.rows = bt.T_max * G;
    p.tile_nodes = kRowTile / G;
    p.tile_rows = p.tile_nodes * G;
    p.g_magic = (65536 + G - 1) / G;
    p.row_tiles = (p.rows + p.tile_rows - 1) / p.tile_rows;
    p.n_layers = n_layers;
    p.z0 = 0;
    p.wait_cycles = knobs.wait_cycles;
    p.withhold = knobs.withhold;
    return p;
}

// The plan of a call that the 128-key kernel takes (attention_plan.cuh); false: the 64-key kernel is faster.
static bool wide_plan(AttnPlan* p, const sd_batch& bt, int dev, int sms, const TestKnobs& knobs) {
    const long long base = (long long)p->n_layers * bt.B * bt.Hkv * p->row_tiles;
    if (!choose_wide(p, base, bt.max_blocks_per_seq, sms, knobs.chunks, [&](int c) { return wide_resident_clusters(dev, sms, c); }))
        return false;
    p->ranked = (bt.B > 1 && bt.B <= 64 && base * p->n_chunks > sms) ? 1 : 0;
    return true;
}

// The others run the 64-key kernel, two CTAs per SM, whose set-up and output overlap the other CTA's tiles.
static void narrow_plan(AttnPlan* plan, const sd_batch& bt, int sms, const TestKnobs& knobs) {
    AttnPlan& p = *plan;
    const int n_layers = p.n_layers;
    // Pick the chunk count that minimises (waves of CTAs) x (key tiles per CTA + fixed cost),
    // two CTAs being resident per SM.  Few waves are counted whole; many waves balance out.
    const int max_tiles = bt.max_blocks_per_seq;
    const int base = n_layers * bt.B * bt.Hkv * p.row_tiles;
    const int slots = 2 * sms;
    int n = 1;
    double best = 1e30;
    for (int c = 1; c <= kMaxChunks && c <= max_tiles; c *= 2) {   // 128 rows split evenly over the chunks
        const double w = (double)base * c / slots;
        double waves = (w <= 4.0) ? (double)((base * c + slots - 1) / slots) : w;
        // Without chunks, and for up to kSplitRounds whole rounds, the CTAs left over after the last whole
        // round go into a launch of their own, with chunks (launch_group): the partial round then costs
        // a fraction of a round.  (Longer launches run under the power cap, where this gained nothing.)
        if (c == 1 && w > 1.0 && base / slots < kSplitRounds) {
            const int rest = base % slots;
            int ct = 1;                                    // chunks of the remainder's launch
            while (2 * ct <= kMaxChunks && 2 * ct <= max_tiles && rest * 2 * ct <= slots) ct *= 2;
            waves = (double)(base / slots) + (rest == 0 ? 0.0 : (ct > 1 ? 1.0 / ct + 0.1 : 1.0));
        }
        // per CTA: its key tiles, a fixed cost of about three tiles, and the in-cluster merge: two to three
        // tiles' worth for clusters of two and four, about eleven for clusters of eight (measured: with
        // eight chunks a launch gains nothing over four unless it saves more than eight tiles per CTA)
        const int merge = (c == 1) ? 0 : (c == 2 ? 2 : (c == 4 ? 3 : 11));
        const double cost = waves * ((max_tiles + c - 1) / c + 3 + merge);
        if (cost < best - 1e-9) { best = cost; n = c; }
    }
    if (knobs.chunks > 0 && knobs.chunks <= max_tiles && (knobs.chunks & (knobs.chunks - 1)) == 0) n = knobs.chunks;     // test hook
    p.set_chunks(n, -1);
    p.tree_blocks = 0;
    p.ranked = (bt.B > 1 && bt.B <= 64 && (long long)base * n > slots) ? 1 : 0;
}

template <int NL>
static sd_status launch_group(const AttnLayers<NL>& layers, int n_layers, const sd_batch& bt, float scale,
                              int32_t* dev_status, cudaStream_t st) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SD_ERR_CUDA;
    const int sms = sm_count(dev);
    const TestKnobs knobs = test_knobs();
    AttnPlan plan = common_plan(bt, n_layers, knobs);
    const int Z = n_layers * bt.B * bt.Hkv;
    if (wide_plan(&plan, bt, dev, sms, knobs)) return launch_wide<NL>(layers, bt, scale, plan, Z, dev_status, st);
    narrow_plan(&plan, bt, sms, knobs);
    // A launch of whole-sequence CTAs that runs for more than one round ends on a partial round, in which
    // the CTAs left over would each work through a whole sequence while most of the GPU idles.  They go
    // into a second launch of the same kernel with the keys split into chunks (a cluster per row tile),
    // so that the remainder also spreads over the SMs and takes a fraction of a round.  (In a ranked
    // launch these are the shortest sequences.)
    const int slots = 2 * sms;
    const long long ctas = (long long)Z * plan.row_tiles;
    if (plan.n_chunks == 1 && ctas > slots && ctas / slots < kSplitRounds && knobs.chunks == 0) {
        const int z_main = (int)((ctas / slots) * slots / plan.row_tiles);
        const int z_rest = Z - z_main;
        int c = 1;
        while (2 * c <= kMaxChunks && 2 * c <= bt.max_blocks_per_seq &&
               (long long)z_rest * plan.row_tiles * 2 * c <= slots) c *= 2;
        if (z_main > 0 && z_rest > 0 && c > 1) {
            const sd_status s = launch_rows1<NL>(layers, bt, scale, plan, z_main, dev_status, st);
            if (s != SD_OK) return s;
            plan.z0 = z_main;
            plan.set_chunks(c, -1);
            return launch_rows1<NL>(layers, bt, scale, plan, z_rest, dev_status, st);
        }
    }
    return launch_rows1<NL>(layers, bt, scale, plan, Z, dev_status, st);
}

// One launch per group of layers: at most kMaxLayersPerLaunch descriptors fit the kernel's
// parameter space and gridDim.z is limited to 65535.
sd_status launch_attention_layers(const sd_batch& bt, const sd_kv_layer* caches, int L,
                                  const void* const* q, const void* const* kt, const void* const* vt,
                                  float scale, void* const* out, float* const* lse,
                                  int32_t* dev_status, cudaStream_t st) {
    const int per_layer_z = bt.B * bt.Hkv;
    if (per_layer_z > 65535) return SD_ERR_UNSUPPORTED;
    int group = 65535 / per_layer_z;
    if (group > kMaxLayersPerLaunch) group = kMaxLayersPerLaunch;
    for (int l0 = 0; l0 < L; l0 += group) {
        const int nl = (L - l0 < group) ? (L - l0) : group;
        if (nl == 1) {
            AttnLayers<1> one;
            if (!fill_layer(&one.l[0], bt, caches[l0], q[l0], kt[l0], vt[l0], out[l0], lse ? lse[l0] : nullptr))
                return SD_ERR_CUDA;
            sd_status s = launch_group<1>(one, 1, bt, scale, dev_status, st);
            if (s != SD_OK) return s;
        } else {
            AttnLayers<kMaxLayersPerLaunch> many;
            for (int i = 0; i < nl; ++i)
                if (!fill_layer(&many.l[i], bt, caches[l0 + i], q[l0 + i], kt[l0 + i], vt[l0 + i], out[l0 + i],
                                lse ? lse[l0 + i] : nullptr))
                    return SD_ERR_CUDA;
            for (int i = nl; i < kMaxLayersPerLaunch; ++i) many.l[i] = many.l[0];
            sd_status s = launch_group<kMaxLayersPerLaunch>(many, nl, bt, scale, dev_status, st);
            if (s != SD_OK) return s;
        }
    }
    return SD_OK;
}

sd_status launch_attention(const sd_batch& bt, const sd_kv_layer& cache, const void* q,
                           const void* kt, const void* vt, float scale, void* out, float* lse,
                           void* ws, size_t ws_bytes, int32_t* dev_status, cudaStream_t st) {
    (void)ws;
    if (ws_bytes < attention_workspace_bytes(bt)) return SD_ERR_WORKSPACE;
    return launch_attention_layers(bt, &cache, 1, &q, &kt, &vt, scale, &out, &lse, dev_status, st);
}

}  // namespace sdv
