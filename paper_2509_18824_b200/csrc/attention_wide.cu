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
// the one O, which works because a row's reference stays where its first scores put it (see kSumLimit): the
// rare tile that raises it is serialised through a per-warp commit barrier that every tile passes anyway.
#include <atomic>
#include "attention_plan.cuh"
#include "attention_wide.cuh"

namespace sdv {

// EARLY: the first K and V copies go in front of everything else that stands between the wait for the kernel ahead and the tile
// loop (bounds check, zeros of unused rows, set-up of the exchange), about 300 cycles.  Calls whose time is latencies and copies
// gain from it (copies_first); in long calls the tile loop, as it is then compiled, is 40 to 80 of 1270 cycles a tile slower.
template <int NL, bool EARLY>
__global__ void __launch_bounds__(kWThreads, 1)
attn_wide_kernel(const __grid_constant__ AttnLayers<NL> layers, const sd_batch bt,
                 const float scale_log2, const AttnPlan plan, int32_t* status) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const WideShared sh(smem);
    uint8_t *const q_smem = sh.q_smem, *const k_smem = sh.k_smem, *const v_smem = sh.v_smem;
    uint64_t *const k_full = sh.k_full, *const v_full = sh.v_full, *const s_full = sh.s_full, *const v_empty = sh.v_empty;
    uint64_t *const p_full = sh.p_full, *const o_full = sh.o_full, *const q_full = sh.q_full, *const x_full = sh.x_full;
    uint32_t* const tmem_slot = sh.tmem_slot;
    int* const abort_flag = sh.abort_flag;
    float *const ref_smem = sh.ref_smem, *const sum_smem = sh.sum_smem;

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
                sh.init_barriers();
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
    const int G = bt.Hq / bt.Hkv;
    const int T = bt.T_max;
    const int tile_rows = plan.tile_rows;
    const uint64_t pol = policy_evict_first();
    // The work of this CTA is worked out before the wait for the kernel ahead, from the length and node count
    // that stand there now, although that kernel may still change them: behind the wait they are read again,
    // and where they differ it is worked out anew.  (Layers of one step find them unchanged.  With all of it
    // behind the wait 2400 cycles passed from there to the first K copy, 700 of them for the reads.  With this and the
    // early report below a call for one sequence of 2048 tokens takes 9.7 instead of 10.5 us, eight chains of
    // 11 nodes over 4096 tokens 16.4 instead of 17.1.)
    int n = 0, len = 0;
    if (!plan.ranked) { n = __ldcg(bt.n_nodes + rank_b); len = __ldcg(bt.len + rank_b); }
    WideWork wk = wide_work(bt, plan, n, len, chunk);
    wk.settle();
    griddep_wait();                                        // global memory from here on

    int b = rank_b;
    if (plan.ranked) b = sequence_of_rank(bt, rank_b, *sh.seq);
    const int32_t *n_nodes = bt.n_nodes, *lens = bt.len, *tables = bt.block_table;
    settle(n_nodes); settle(lens); settle(tables);         // (no load of theirs in front of the wait)
    // (lengths that a kernel of this library wrote while this one was already there: not for the read-only path)
    const int32_t* const seq_table = tables + (size_t)b * bt.max_blocks_per_seq;
    const int n_now = __ldcg(n_nodes + b), len_now = __ldcg(lens + b);
    int even = 0, odd = 0;                                 // block table of this chunk (producer warp)
    if (warp == kWTmaWarp) {
        const int i = wk.t0 + lane;                        // (within the table whatever the length)
        if (i < bt.max_blocks_per_seq) even = __ldg(seq_table + i);
        if (i + 32 < bt.max_blocks_per_seq) odd = __ldg(seq_table + i + 32);
        if (aligned && lane == 0) {                        // Q depends on nothing but b
            mbar_arrive_expect_tx(q_full, (uint32_t)tile_rows * kD * 2);
            tma_load_3d(q_smem, &ly.q, 0, kvh * G, b * T + rt * plan.tile_nodes, q_full, pol);
            tma_load_3d(q_smem + kRowTile * 128, &ly.q, 64, kvh * G, b * T + rt * plan.tile_nodes, q_full, pol);
        }
        __syncwarp();
    }
    const bool as_guessed = n_now == n && len_now == len;
    const int t0_read = wk.t0;                             // where `even` and `odd` were read
    if (!as_guessed) wk = wide_work(bt, plan, n_now, len_now, chunk);
    n = wk.n; len = wk.len;
    const int rows = n * G;                                // rows of this sequence's own nodes
    const bool m64 = (rows - rt * tile_rows) <= 64;        // last row tile of at most 64 rows: M = 64 (lanes 0..15 of a quadrant)
    auto check_length = [&] {
        if ((len + kBlock - 1) / kBlock > bt.max_blocks_per_seq && threadIdx.x == 0) set_status(status, SD_ERR_BOUNDS);
    };
    if constexpr (!EARLY) check_length();
    const int n_chunks = wk.n_chunks, n_pref = wk.n_pref, nb = wk.nb, t0 = wk.t0;
    const int nt = (nb + 1) / 2;
    const bool has_rows = rt * tile_rows < rows && chunk < n_chunks;   // (CTAs beyond have nothing to do)
    const bool active = (nt > 0) && aligned && has_rows;
    const bool clustered = (n_chunks > 1) && has_rows;     // (a CTA without work leaves; cluster barriers do not wait for it)
    const int32_t* table = seq_table + t0;
    // The producer is a whole warp in uniform control flow with one lane elected around the copies (32 cycles
    // per copy; 70 from a lane-0 branch, where every operand has to be moved to uniform registers under
    // divergence, and eight copies a tile made the producer the kernel's bound).  Its lanes hold the
    // block table: 32 entries in `even` (blocks 64 w ..) and 32 in `odd` (blocks 64 w + 32 ..), fetched a
    // window ahead, handed out by shuffles.
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
    auto first_copies = [&] {
        if (t0 != t0_read) {
            even = window(0);
            odd = window(32);
        }
#pragma unroll
        for (int i = 0; i < kWStages; ++i)
            if (i < nt) {
                issue(i, i, false);
                issue(i, i, true);
            }
    };
    if constexpr (EARLY) {
        if (active && warp == kWTmaWarp) first_copies();
        check_length();
        if (chunk == 0 && warp < 8) zero_unused_rows(bt, plan, ly, b, rt, kvh, rows, (int)threadIdx.x, 256);
    } else {
        if (chunk == 0) zero_unused_rows(bt, plan, ly, b, rt, kvh, rows, (int)threadIdx.x, kWThreads);
    }
    float m_used = -INFINITY, l = 0.f;                     // this thread's row: reference, sum over its group's tiles
    bool rows_ready = false;
    const RowExchange x{bt, plan, ly, smem_u32(k_smem), smem_u32(x_full), chunk, n_chunks, rt, b, kvh, rows, wk.tpc, wk.tiles_total};
    // The chunks' rows meet in the K ring as described at RowExchange.  A CTA's K ring is free when its last scores
    // are there, which is where its warps report it to the cluster: the barrier then hides behind the last
    // tile's exponentials and P.V (reported behind them it took another 850 cycles).
    if (clustered && warp == kWMmaWarp && lane == 0) exchange_expect(x, x_full);
    auto ring_is_free = [&] {
        __syncwarp();
        if (clustered) cluster_arrive_release();
    };

    if (active) {
    if (warp == kWTmaWarp) {
        // ------------------------------------------------------------ TMA producer
        if constexpr (!EARLY) first_copies();
        int jk = min(nt, kWStages), jv = jk;
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
            unwind_pause();
        }
        ring_is_free();
    } else if (warp == kWMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        const int M = m64 ? 64 : kRowTile;
        const uint32_t idesc_s = make_idesc_bf16(M, kWTile, false, false), idesc_s_half = make_idesc_bf16(M, kWTile / 2, false, false);
        const uint32_t idesc_o = make_idesc_bf16(M, kD, false, true);
        // (A whole warp in uniform control flow, one lane elected around the instructions, as in the producer: eight
        //  MMAs take 375 to 440 cycles to issue; a warp of one thread needed 470 to 480.)
        const uint64_t qdesc = make_smem_desc(smem_u32(q_smem), 16, 1024, 128);
        const uint64_t kdesc0 = make_smem_desc(smem_u32(k_smem), 16, 1024, 128);
        const uint64_t vdesc0 = make_smem_desc(smem_u32(v_smem), kWHalf, 1024, 128);   // [key][d]: N (= d) contiguous
        bool ok = mbar_wait_warp(q_full, 0, abort_flag, plan.wait_cycles);
        auto issue_s = [&](int j) -> bool {
            const int s = j % kWStages;
            if (!mbar_wait_warp(&k_full[s], (uint32_t)(j / kWStages) & 1u, abort_flag, plan.wait_cycles)) return false;
            tc_fence_after_sync();
            const uint64_t kd = kdesc0 + (uint64_t)(s * (kWStage >> 4));
            const uint32_t d = tmem_s + s * kWTile;
            const uint32_t idesc = 2 * j + 1 < nb ? idesc_s : idesc_s_half;
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < kD / 16; ++k)
                    mma_ss(d, qdesc + (uint64_t)((k >> 2) * ((kRowTile * 128) >> 4) + (k & 3) * 2),
                           kd + (uint64_t)((k >> 2) * (kWHalf >> 4) + (k & 3) * 2), idesc, k != 0 ? 1u : 0u);
                mma_commit(&s_full[s]);
            }
            __syncwarp();
            return true;
        };
        for (int j = 0; j < kWStages - 1 && j < nt && ok; ++j) ok = issue_s(j);
        for (int j = 0; j < nt && ok; ++j) {
            // scores two tiles ahead: their buffer held P of tile j - 1, whose P.V was issued before
            if (j + kWStages - 1 < nt) ok = issue_s(j + kWStages - 1);
            if (!ok) break;
            const int s = j % kWStages;
            const uint32_t ph = (uint32_t)(j / kWStages) & 1u;
            if (!mbar_wait_warp(&p_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
            if (!mbar_wait_warp(&v_full[s], ph, abort_flag, plan.wait_cycles)) { ok = false; break; }
            tc_fence_after_sync();
            const uint64_t vd = vdesc0 + (uint64_t)(s * (kWStage >> 4));
            const uint32_t pa = tmem_s + s * kWTile;       // P from tensor memory: 16 keys = 8 columns
            const uint32_t first = (j != 0) ? 1u : 0u;
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    mma_ts(tmem_o, pa + k * 8, vd + (uint64_t)(k * (2048 >> 4)), idesc_o, k != 0 ? 1u : first);
                if (2 * j + 1 < nb) {
#pragma unroll
                    for (int k = 4; k < 8; ++k) mma_ts(tmem_o, pa + k * 8, vd + (uint64_t)(k * (2048 >> 4)), idesc_o, 1u);
                }
                mma_commit(&v_empty[s]);
            }
            __syncwarp();
        }
        if (elect_one()) mma_commit(o_full);
        __syncwarp();
        if (!ok) {
            // unwinding: nothing may give tensor memory back while an MMA issued above still runs
            if (lane == 0) set_status(status, SD_ERR_TIMEOUT);
            mbar_wait_plain(o_full, 0, plan.wait_cycles);
            unwind_pause();
        }
        ring_is_free();
    } else {
        // ------------------------------------------------------------ softmax: one thread per row and group
        const int group = warp >> 2, quad = warp & 3;
        const int gt = quad * 32 + lane;                   // TMEM lane, also the index within the group
        const int row_in_tile = m64 ? (lane < 16 ? quad * 16 + lane : -1) : gt;    // -1: a TMEM lane without a row
        const int row = (row_in_tile >= 0 && row_in_tile < tile_rows) ? rt * tile_rows + row_in_tile : rows;
        const bool row_ok = row < rows;
        const uint64_t amask = row_ok ? bt.anc_mask[(size_t)b * T + plan.node_of(row)] : ~0ull;
        const uint32_t lane_field = (uint32_t)(quad * 32) << 16;
        bool ok = wide_softmax(plan, sh, WideTiles{nt, nb, n_pref, t0, len, n}, tmem_o, tmem_s, group, quad, lane, row_ok, amask,
                               scale_log2, m_used, l);
        ring_is_free();
        volatile float* my_ref = ref_smem + gt;
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
        } else {
            if (lane == 0) set_status(status, SD_ERR_TIMEOUT);
            unwind_pause();
        }
    }
    } else {
        ring_is_free();
    }

    if (!active && aligned && warp == kWTmaWarp && lane == 0 && !mbar_wait(q_full, 0, abort_flag, plan.wait_cycles)) {   // nobody else waits for the Q copy
        set_status(status, SD_ERR_TIMEOUT);
        unwind_pause();
    }

    if (clustered) {
        const int gt = (int)threadIdx.x & 127;
        const int row_in_tile = m64 ? (lane < 16 ? (warp & 3) * 16 + lane : -1) : gt;
        __syncwarp();
        cluster_wait_acquire();                            // every chunk's K ring is free
        if (active && warp < 8)
            exchange_push<2>(x, tmem_base + ((uint32_t)((warp & 3) * 32) << 16), (warp >> 2) * 2, rows_ready, row_in_tile, m_used, l);
        __syncwarp();
        cluster_arrive_relaxed();                          // (waited for at the end: nobody leaves before its peers have sent)
        bool late = false;
        if (warp < 8) {
            asm volatile("bar.sync 1, 256;" ::: "memory"); // this CTA's own rows
            if (mbar_wait_cluster(x_full, 0, abort_flag, plan.wait_cycles)) {
                switch (n_chunks) {
                    case 2: merge_rows<2, 256>(x, (int)threadIdx.x); break;
                    case 3: merge_rows<3, 256>(x, (int)threadIdx.x); break;
                    case 4: merge_rows<4, 256>(x, (int)threadIdx.x); break;
                    case 5: merge_rows<5, 256>(x, (int)threadIdx.x); break;
                    case 6: merge_rows<6, 256>(x, (int)threadIdx.x); break;
                    case 7: merge_rows<7, 256>(x, (int)threadIdx.x); break;
                    default: merge_rows<8, 256>(x, (int)threadIdx.x); break;
                }
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
    if (warp == kWTmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

template <int NL>
sd_status launch_wide(const AttnLayers<NL>& layers, const sd_batch& bt, float scale, const AttnPlan& plan,
                      int z_count, int32_t* dev_status, cudaStream_t st) {
    if constexpr (NL == 1)
        if (copies_first(plan, bt.max_blocks_per_seq))
            return launch_attn(attn_wide_kernel<NL, true>, kWThreads, kWSmem, layers, bt, scale, plan, z_count, dev_status, st);
    return launch_attn(attn_wide_kernel<NL, false>, kWThreads, kWSmem, layers, bt, scale, plan, z_count, dev_status, st);
}
template sd_status launch_wide<1>(const AttnLayers<1>&, const sd_batch&, float, const AttnPlan&, int, int32_t*, cudaStream_t);
template sd_status launch_wide<kMaxLayersPerLaunch>(const AttnLayers<kMaxLayersPerLaunch>&, const sd_batch&, float,
                                                    const AttnPlan&, int, int32_t*, cudaStream_t);

// Clusters of n_chunks CTAs that the current device runs at a time (asked once per device and size: with one
// CTA per SM it depends on how many SMs each GPC has; 8 x 16 of the 148 do not all fit, for instance).
int wide_resident_clusters(int dev, int sms, int n_chunks) {
    constexpr int kDevs = 64;
    static std::atomic<int> cache[kDevs][kMaxChunks + 1];
    if (n_chunks <= 1) return sms;
    if (dev >= 0 && dev < kDevs)
        if (const int v = cache[dev][n_chunks].load(std::memory_order_relaxed)) return v;
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
    if (cudaFuncSetAttribute(attn_wide_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, attn_wide_kernel<1, false>, &cfg) != cudaSuccess || n < 1)
        n = max(1, sms / n_chunks - n_chunks);             // (no answer: a cautious guess, and ask again next time)
    else if (dev >= 0 && dev < kDevs)
        cache[dev][n_chunks].store(n, std::memory_order_relaxed);
    return n;
}

}  // namespace sdv
