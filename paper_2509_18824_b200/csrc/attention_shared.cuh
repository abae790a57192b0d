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
constexpr int kMaxChunks = 8;                  // = portable cluster size
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
__device__ __forceinline__ void mask_scores(uint32_t (&r)[32], uint32_t mask) {
#pragma unroll
    for (int c = 0; c < 32; ++c) r[c] = ((mask >> c) & 1u) ? r[c] : 0xff800000u;
}

// 32 raw scores of a row -> 2^(score * scale - reference), packed to bf16 in pairs, and added to the sums
__device__ __forceinline__ void exp_pack_half(const uint32_t (&r)[32], uint64_t scale2, uint64_t neg_m2, uint32_t* pk,
                                              uint64_t (&ps)[2]) {
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const uint64_t x = fma_f32x2(pack_f32x2(__uint_as_float(r[2 * c]), __uint_as_float(r[2 * c + 1])), scale2, neg_m2);
        float x0, x1;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x));
        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
        ps[c & 1] = add_f32x2(ps[c & 1], pack_f32x2(p0, p1));
        const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
        pk[c] = *reinterpret_cast<const uint32_t*>(&h);
    }
}

struct AttnPlan {
    int n_chunks;      // key chunks per sequence (the last one also takes the tree tile)
    int rows;          // T_max * G
    int tile_nodes;    // tree nodes of a row tile: its rows are whole nodes, the query heads of one KV head each
    int tile_rows;     // tile_nodes * G <= 128
    int row_tiles;
    int n_layers;      // layers of this launch
    int ranked;        // dispatch the sequences longest first (only matters when the grid runs in several waves)
    int z0;            // first (sequence rank, layer, KV head) index of this launch: blockIdx.z counts from here
    long long wait_cycles;   // bound of every barrier wait, in SM cycles
    int withhold;      // test hook: the softmax warps never report their first tile, so that a wait runs out
};

// cache blocks [t0, t1) of one key chunk of a sequence
struct ChunkRange { int tiles_total, tpc, t0, t1; };
__device__ __forceinline__ ChunkRange chunk_range(int len, int max_blocks, int n_chunks, int chunk) {
    ChunkRange r;
    r.tiles_total = min((len + kBlock - 1) / kBlock, max_blocks);
    r.tpc = (r.tiles_total + n_chunks - 1) / n_chunks;
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

// Final step of a clustered launch.  The CTA of chunk o finishes rows o * 128 / NCH .. of the tile and
// holds, in its exchange area, those rows' unnormalised O of every chunk ([chunk][16-byte piece][row], its
// own rows stored locally, the others' by the CTAs that computed them) and their references and sums
// ([chunk][row] each).  One thread takes one row and 16 output columns at a time: consecutive lanes read
// consecutive rows of a piece (no bank conflicts) and each writes a whole 32-byte sector; chunks are
// added in chunk order, so the result does not depend on timing.
struct MergeCtx {
    const sd_batch& bt; const AttnPlan& plan; __nv_bfloat16* out; float* lse;
    uint32_t xo_addr, xs_addr;          // this CTA's exchange area: rows, then references [128] and sums [128]
    int chunk, rt, b, kvh, rows, tpc, tiles_total, tid;
};

template <int NCH>
__device__ __forceinline__ void merge_rows(const MergeCtx& x) {
    constexpr int kRowsPer = kRowTile / NCH;        // rows this CTA finishes
    const int G = x.bt.Hq / x.bt.Hkv;
    const int rl = x.tid % kRowsPer;
    const int in_tile = x.chunk * kRowsPer + rl, row = x.rt * x.plan.tile_rows + in_tile;
    if (in_tile >= x.plan.tile_rows || row >= x.rows) return;      // only rows of the sequence were sent
    float w[NCH];
    float M = -INFINITY;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const bool live = (c == NCH - 1) || (c * x.tpc < x.tiles_total);       // that chunk had key tiles
        w[c] = live ? ld_smem_f32(x.xs_addr + (c * kRowsPer + rl) * 4) : -INFINITY;
        M = fmaxf(M, w[c]);
    }
    float den = 0.f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        if (w[c] == -INFINITY) { w[c] = 0.f; continue; }
        w[c] = ex2_approx(w[c] - M);
        den = fmaf(w[c], ld_smem_f32(x.xs_addr + (kRowTile + c * kRowsPer + rl) * 4), den);
    }
    const float inv = __frcp_rn(den);
    const int node = row / G, g = row - node * G;
    const size_t orow = ((size_t)x.b * x.bt.T_max + node) * x.bt.Hq + x.kvh * G + g;
    if (x.lse && x.tid < kRowsPer) x.lse[orow] = (M + __log2f(den)) * 0.6931471805599453f;
#pragma unroll
    for (int cg = x.tid / kRowsPer; cg < 8; cg += kRowTile / kRowsPer) {       // 16 columns: pieces 4 cg .. + 3
        float4 acc[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            if (!((c == NCH - 1) || (c * x.tpc < x.tiles_total))) continue;    // (nothing was written there)
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
        uint4* dst = reinterpret_cast<uint4*>(x.out + orow * kD + cg * 16);
        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// one launch of `z_count` (sequence rank, layer, KV head) groups starting at plan.z0
template <int NL>
sd_status launch_rows1(const AttnLayers<NL>& layers, const sd_batch& bt, float scale, const AttnPlan& plan,
                       int z_count, int32_t* dev_status, cudaStream_t st);     // one row tile per CTA, 64-key tiles

}  // namespace sdv
