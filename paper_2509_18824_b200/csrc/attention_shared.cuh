// Pieces of the tree-attention kernel that its launcher shares with it: launch plan, per-layer
// descriptors, and the in-cluster merge of key chunks through distributed shared memory.
#pragma once
#include <stdlib.h>
#include "common.cuh"
#include "sm100.cuh"

namespace sdv {
using namespace sm100;

constexpr int kRowTile = 128;                  // query rows per row tile (MMA M)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kSumLimit = 1.0995e12f;        // 2^40: a tile's sum above this raises the row's reference
constexpr float kRaiseAbove = 32.f;            // log2 units: ... where the maximum itself is looked at (128 x 2^32 < 2^40)
constexpr int kMaxChunks = 8;                  // = portable cluster size
constexpr int kStartBlocks = 5;                // cache blocks that fit the 128-key kernel's ring at once beside the tree's
constexpr int kTreeBlocks = 3;                 // blocks that the tree counts for in longer chunks, see chunk_range
constexpr int kSplitRounds = 8;                // launches of fewer whole rounds get their remainder as a chunked launch

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// two fp32 values per 64-bit register: one instruction scales, or adds, both (round to nearest even, each)
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float sum_f32x2(uint64_t a) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
    return lo + hi;
}

// keys outside the mask get the score -inf
template <int N>
__device__ __forceinline__ void mask_scores(uint32_t (&r)[N], uint32_t mask) {
#pragma unroll
    for (int c = 0; c < N; ++c) r[c] = ((mask >> c) & 1u) ? r[c] : 0xff800000u;
}

// N raw scores of a row -> 2^(score * scale - reference), packed to bf16 in pairs, and added to the sums
template <int N>
__device__ __forceinline__ void exp_pack(const uint32_t (&r)[N], uint64_t scale2, uint64_t neg_m2, uint32_t* pk,
                                              uint64_t (&ps)[2]) {
#pragma unroll
    for (int c = 0; c < N / 2; ++c) {
        const uint64_t x = fma_f32x2(pack_f32x2(__uint_as_float(r[2 * c]), __uint_as_float(r[2 * c + 1])), scale2, neg_m2);
        float x0, x1;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x));
        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
        ps[c & 1] = add_f32x2(ps[c & 1], pack_f32x2(p0, p1));
        const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
        pk[c] = *reinterpret_cast<const uint32_t*>(&h);
    }
}

// rows of a row tile that each of its chunks' CTAs finishes: in eights, so that what a warp sends to one CTA
// are whole 128-byte lines (the last CTAs may have fewer, or none)
__host__ __device__ constexpr int rows_per_chunk(int n_chunks) { return ((kRowTile + n_chunks - 1) / n_chunks + 7) & ~7; }

struct AttnPlan {
    int n_chunks;      // CTAs per row tile along the keys (a cluster): the most chunks that a sequence's keys are cut into
    int whole_blocks;  // sequences of at most so many cache blocks stay whole; -1: every one is cut into n_chunks
    int tree_blocks = 0;     // cache blocks that the tree's keys count for in chunks of more than kStartBlocks (chunk_range)
    uint32_t chunk_magic;    // ceil(2^32 / n_chunks): x / n_chunks for x below 2^29 (n_chunks > 1)
    int rows;          // T_max * G
    int tile_nodes;    // tree nodes of a row tile: its rows are whole nodes, the query heads of one KV head each
    int tile_rows;     // tile_nodes * G <= 128
    int row_tiles;
    int g_magic;       // ceil(65536 / G): row / G for rows below 64 * 8
    __host__ __device__ __forceinline__ int node_of(int row) const { return (row * g_magic) >> 16; }
    void set_chunks(int n, int whole) { n_chunks = n; whole_blocks = whole; chunk_magic = (uint32_t)((0x100000000ull + n - 1) / n); }
    int n_layers;      // layers of this launch
    int ranked;        // dispatch the sequences longest first (only matters when the grid runs in several waves)
    int z0;            // first (sequence rank, layer, KV head) index of this launch: blockIdx.z counts from here
    long long wait_cycles;   // bound of every barrier wait, in SM cycles
    int withhold;      // test hook: the softmax warps never report their first tile, so that a wait runs out
};

// blockIdx.z enumerates (sequence rank, layer, KV head): the CTAs of the longest sequences are dispatched
// first, in every layer, so that a ragged batch does not end on a few long stragglers.  The rank -> sequence
// lookup is done here (up to 64 sequences: each of the first B threads ranks one sequence by cached length,
// ties by index); larger batches, and launches that fit the GPU in one round, run in index order.
__device__ __forceinline__ int sequence_of_rank(const sd_batch& bt, int rank, int& s_seq) {
    const int32_t* lens = bt.len;
    settle(lens);
    if ((int)threadIdx.x < bt.B) {
        const int mine = __ldcg(lens + threadIdx.x);
        int r = 0;
        for (int j = 0; j < bt.B; ++j) {
            const int other = __ldcg(lens + j);
            r += (other > mine || (other == mine && j < (int)threadIdx.x)) ? 1 : 0;
        }
        if (r == rank) s_seq = threadIdx.x;
    }
    __syncthreads();
    return s_seq;
}

// The key chunks of a sequence (the last one also takes the tree's keys), and the cache blocks [t0, t1) of one of them.
// Where sequences may stay whole, the others are cut into the smallest number of chunks, up to n_chunks, whose longest
// is as short as n_chunks make it.  All of it follows from the sequence's own length: the block table may be far
// wider than any sequence of the batch.
// The tree's keys, in the last chunk, take as long as about three blocks where their copies cannot start with the first
// ones (kStartBlocks and the tree fill the ring): they wait for a V slot, the softmax for them, because it clears the
// rows of unused nodes, and masked scores take longer.  With the blocks alone dealt out evenly the last chunk's
// softmax ended 1.6 us behind the others' of one sequence of 2048 tokens and 60 nodes, 3 us in eight chains of 4096
// tokens.  Us per call with the tree counted as 0, 1, 2, 3, 4 blocks: eight chains of 4096 tokens 16.8 16.4 16.4 16.4
// 16.4, four sequences of 2048 and 60 nodes 13.9 14.3 14.4 14.0 14.0, one chain of 8192 13.1 12.6 12.6 12.6 12.6, 28 layers
// of one sequence of 2048 (and the LM head) 468 456 456 456 456; in shorter chunks it gains nothing (15 blocks in four
// chunks: 8.05 8.17 9.01 9.04 8.97: an odd block is half a tile).  Nor does it where the even split leaves the last chunk four
// blocks or fewer, which with the tree are no more than the others have: two sequences of 1369 tokens and 55 nodes (22 blocks in
// four, 6 6 6 4 or 7 7 7 1) 9.85 and 10.74, five such splits 2 to 7 % slower.  Over 436 splits with a longer last
// chunk (trees of 2 to 64 nodes, 1 to 16 sequences) three blocks against none are 2.7 % faster on average, 10 % at best; 5 %
// slower at worst.  Where a boundary lies also decides the scores that a chunk's reference comes
// from, and so where P rounds to bf16: with other boundaries outputs differ by about 2.5e-3 relative, no more than either is
// from fp64 (2.295e-3 on average over twelve sequences of 2048 to 3148 tokens evenly split, 2.293e-3 so).
struct ChunkRange { int n_chunks, tiles_total, tpc, t0, t1; };
__host__ __device__ __forceinline__ ChunkRange chunk_range(const AttnPlan& plan, int len, int max_blocks, int chunk) {
    ChunkRange r;
    r.tiles_total = min((len + kBlock - 1) / kBlock, max_blocks);
    const bool whole = plan.n_chunks == 1 || r.tiles_total <= max(plan.whole_blocks, 0);
    const auto share = [&](int blocks) { return (int)(((uint64_t)(uint32_t)(blocks + plan.n_chunks - 1) * plan.chunk_magic) >> 32); };
    const int even = share(r.tiles_total), behind = r.tiles_total - (plan.n_chunks - 1) * even;
    const int last = behind > 0 ? behind : behind + even;      // (more than kStartBlocks each: at most one chunk stays empty)
    const int counted = r.tiles_total + (even > kStartBlocks && last >= kStartBlocks ? plan.tree_blocks : 0);
    r.tpc = whole ? r.tiles_total : share(counted);
    r.n_chunks = whole ? 1 : plan.n_chunks;
    if (plan.whole_blocks >= 0 && !whole) {
        r.n_chunks = 2;
        while (r.n_chunks * r.tpc < counted) ++r.n_chunks;
    }
    r.t0 = min(chunk * r.tpc, r.tiles_total);
    r.t1 = min(r.t0 + r.tpc, r.tiles_total);
    return r;
}

// Everything the CTAs of one layer need.  A launch covers up to kMaxLayersPerLaunch layers (the
// descriptors travel as kernel parameters); blockIdx.z enumerates (sequence, layer, KV head).
struct AttnLayer {
    CUtensorMap q;                  // 3-D (128, Hq, B*T_max), box 64 x G x tile_nodes
    CUtensorMap k_cache, v_cache;   // 2-D [num_blocks*Hkv*64][128], box 64 x 64
    CUtensorMap k_tree, v_tree;     // 3-D (128, Hkv, B*T_max), box 64 x 1 x 64
    __nv_bfloat16* out;             // bf16 [B][T_max][Hq][D]
    float* lse;                     // f32  [B][T_max][Hq] or null
    int32_t num_blocks;
};
constexpr int kMaxLayersPerLaunch = 32;
template <int NL>
struct AttnLayers { AttnLayer l[NL]; };

// rows of unused nodes become zeros, 16 bytes per thread (by the CTA of the first chunk)
__device__ __forceinline__ void zero_unused_rows(const sd_batch& bt, const AttnPlan& plan, const AttnLayer& ly, int b, int rt, int kvh,
                                                 int rows, int tid, int threads) {
    const int G = bt.Hq / bt.Hkv;
    const int z0 = max(rows, rt * plan.tile_rows), z1 = min(plan.rows, (rt + 1) * plan.tile_rows);
    for (int i = z0 * 16 + tid; i < z1 * 16; i += threads) {
        const int row = i >> 4, node = plan.node_of(row);
        const size_t orow = ((size_t)b * bt.T_max + node) * bt.Hq + kvh * G + (row - node * G);
        reinterpret_cast<uint4*>(ly.out + orow * kD)[i & 15] = make_uint4(0, 0, 0, 0);
        if (ly.lse && (i & 15) == 0) ly.lse[orow] = 0.f;
    }
}

// Final step of a clustered launch.  Row r of the tile is finished by the CTA of chunk r / rows_per_chunk.
// Every other chunk's CTA sends it that row's reference, sum and unnormalised O straight from tensor memory,
// with stores that report their bytes to the receiver's barrier (so the receiver waits for exactly what it
// gets, and no second cluster-wide barrier and release stand between the last row and the merge); its own
// rows it stores locally.
// Exchange area (over the K ring): [chunk][16-byte piece of the row][row of the finisher], so that a warp's
// store (32 rows, one piece each) fills 512 consecutive bytes: remote stores travel in packets of
// consecutive bytes (measured with 256 CTAs in pairs: 24.5 B/clk per CTA against 12.5 for one 512-byte
// line per row); behind it references and sums, [chunk][row] each.
struct RowExchange {
    const sd_batch& bt; const AttnPlan& plan; const AttnLayer& ly;
    uint32_t xo_addr;                   // this CTA's exchange area
    uint32_t bar_addr;                  // its barrier for the rows of the other chunks
    int chunk, n_chunks, rt, b, kvh, rows, tpc, tiles_total;
    __device__ __forceinline__ uint32_t sum_off() const { return (uint32_t)(n_chunks * rows_per_chunk(n_chunks)) * 4; }
    __device__ __forceinline__ uint32_t xs_addr() const { return xo_addr + sum_off() * kD; }
    // rows beyond the sequence's last one are not exchanged
    __device__ __forceinline__ bool has(int in_tile) const { return in_tile < plan.tile_rows && rt * plan.tile_rows + in_tile < rows; }
    // does that chunk have key tiles (the last one has the tree's)
    __device__ __forceinline__ bool live(int c) const { return c == n_chunks - 1 || c * tpc < tiles_total; }
};

// bytes this CTA will receive (one thread, before the cluster barrier)
__device__ __forceinline__ void exchange_expect(const RowExchange& x, uint64_t* bar) {
    const int per = rows_per_chunk(x.n_chunks);
    const int mine = min(max(min(x.rows - x.rt * x.plan.tile_rows, x.plan.tile_rows) - x.chunk * per, 0), per);
    int others = 0;
    for (int c = 0; c < x.n_chunks; ++c) others += (c != x.chunk && x.live(c)) ? 1 : 0;
    mbar_arrive_expect_tx(bar, (uint32_t)(others * mine * (kD * 4 + 8)));
}

// NC 32-column pieces of this thread's row from column 32 * cc0 on; tmem: O at this warp's lanes
template <int NC>
__device__ __forceinline__ void exchange_push(const RowExchange& x, uint32_t tmem, int cc0, bool ready, int row_in_tile, float ref,
                                              float sum) {
    const int per = rows_per_chunk(x.n_chunks);
    const int rr = max(row_in_tile, 0), dest = rr / per, rl = rr - dest * per;
    const bool mine = ready && row_in_tile >= 0 && x.has(rr), remote = dest != x.chunk;
    const uint32_t off = (uint32_t)((x.chunk * 32 * per + rl) * 16);
    const uint32_t xo = (remote ? map_dsmem(x.xo_addr, (uint32_t)dest) : x.xo_addr) + off;
    const uint32_t bar = map_dsmem(x.bar_addr, (uint32_t)dest);
    tc_fence_after_sync();
#pragma unroll
    for (int cc = cc0; cc < cc0 + NC; ++cc) {
        uint32_t o[32];
        tmem_ld32(tmem + cc * 32, o);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t at = xo + (uint32_t)((cc * 8 + k) * per * 16);
            if (mine && remote) st_async_v4(at, o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3], bar);
            else if (mine) st_smem_v4(at, o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
        }
    }
    if (mine && cc0 == 0) {
        const uint32_t at = x.xs_addr() + (uint32_t)(x.chunk * per + rl) * 4;
        if (remote) {
            const uint32_t to = map_dsmem(at, (uint32_t)dest);
            st_async_b32(to, __float_as_uint(ref), bar);
            st_async_b32(to + x.sum_off(), __float_as_uint(sum), bar);
        } else {
            st_smem_f32(at, ref);
            st_smem_f32(at + x.sum_off(), sum);
        }
    }
}

// The finisher adds up the chunks in chunk order (so the result does not depend on timing).  One thread takes
// one row and 16 output columns at a time: consecutive lanes read consecutive rows of a piece (no bank
// conflicts) and each writes a whole 32-byte sector.
template <int NCH, int THREADS>
__device__ __forceinline__ void merge_rows(const RowExchange& x, int tid) {
    constexpr int kRowsPer = rows_per_chunk(NCH);   // rows this CTA finishes
    constexpr int kGroups = THREADS / kRowsPer;     // threads that share a row (those beyond the last whole group rest)
    const int G = x.bt.Hq / x.bt.Hkv;
    const int rl = tid % kRowsPer;
    const int in_tile = x.chunk * kRowsPer + rl, row = x.rt * x.plan.tile_rows + in_tile;
    if (tid >= kGroups * kRowsPer || !x.has(in_tile)) return;
    const uint32_t xs = x.xo_addr + NCH * kRowsPer * kD * 4;
    float w[NCH];
    float M = -INFINITY;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        w[c] = x.live(c) ? ld_smem_f32(xs + (c * kRowsPer + rl) * 4) : -INFINITY;
        M = fmaxf(M, w[c]);
    }
    float den = 0.f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        if (w[c] == -INFINITY) { w[c] = 0.f; continue; }
        w[c] = ex2_approx(w[c] - M);
        den = fmaf(w[c], ld_smem_f32(xs + (NCH * kRowsPer + c * kRowsPer + rl) * 4), den);
    }
    const float inv = __frcp_rn(den);
    const int node = x.plan.node_of(row), g = row - node * G;
    const size_t orow = ((size_t)x.b * x.bt.T_max + node) * x.bt.Hq + x.kvh * G + g;
    if (x.ly.lse && tid < kRowsPer) x.ly.lse[orow] = (M + __log2f(den)) * 0.6931471805599453f;
#pragma unroll
    for (int cg = tid / kRowsPer; cg < 8; cg += kGroups) {       // 16 columns: pieces 4 cg .. + 3
        float4 acc[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            if (!x.live(c)) continue;                                  // (nothing was written there)
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float4 v = ld_smem_v4(x.xo_addr + (uint32_t)(((c * 32 + cg * 4 + p) * kRowsPer + rl) * 16));
                acc[p].x = fmaf(w[c], v.x, acc[p].x); acc[p].y = fmaf(w[c], v.y, acc[p].y);
                acc[p].z = fmaf(w[c], v.z, acc[p].z); acc[p].w = fmaf(w[c], v.w, acc[p].w);
            }
        }
        uint32_t o[8];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const __nv_bfloat162 h0 = __floats2bfloat162_rn(acc[p].x * inv, acc[p].y * inv);
            const __nv_bfloat162 h1 = __floats2bfloat162_rn(acc[p].z * inv, acc[p].w * inv);
            o[2 * p] = *reinterpret_cast<const uint32_t*>(&h0);
            o[2 * p + 1] = *reinterpret_cast<const uint32_t*>(&h1);
        }
        uint4* dst = reinterpret_cast<uint4*>(x.ly.out + orow * kD + cg * 16);
        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// one launch of `z_count` (sequence rank, layer, KV head) groups starting at plan.z0
template <typename Kernel, typename Layers>
sd_status launch_attn(Kernel kern, int threads, int smem, const Layers& layers, const sd_batch& bt, float scale,
                      const AttnPlan& plan, int z_count, int32_t* dev_status, cudaStream_t st) {
    if (!allow_dynamic_smem(kern, smem)) return SD_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.n_chunks, plan.row_tiles, z_count);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;      // the chunks of one row tile form a cluster
    attr[0].val.clusterDim.x = plan.n_chunks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // The launch may begin while the kernel before it in the stream is still running (its CTAs take the
    // SM slots that one frees and do their set-up); the kernel waits for that kernel's completion before
    // it touches global memory.  Consecutive attention calls - one per layer - overlap their ends this way.
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cuda_ok(cudaLaunchKernelEx(&cfg, kern, layers, bt, scale * kLog2e, plan, dev_status));
}
template <int NL>
sd_status launch_rows1(const AttnLayers<NL>& layers, const sd_batch& bt, float scale, const AttnPlan& plan,
                       int z_count, int32_t* dev_status, cudaStream_t st);     // 64-key tiles, two CTAs per SM
template <int NL>
sd_status launch_wide(const AttnLayers<NL>& layers, const sd_batch& bt, float scale, const AttnPlan& plan,
                      int z_count, int32_t* dev_status, cudaStream_t st);      // 128-key tiles, one CTA per SM
int wide_resident_clusters(int dev, int sms, int n_chunks);

}  // namespace sdv
