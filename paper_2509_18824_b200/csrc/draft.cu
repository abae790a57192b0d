// Draft-side target-feature aggregation (Sec. 3.1.1 of the paper): Q meta queries, shared by all
// tokens, attend over the L target-layer features of each token; the core of that cross-attention
// for head size 128.  Streaming work: every token's K and V rows (L x D each) are read once, so the
// roofline is HBM bandwidth.  One warp per (token, head).  The two tiny products (Q x 128 x L and
// Q x L x 128, Q <= 8) run as warp-level mma.sync m16n8k16 (rows 8..15 of the A operands are zero):
// with scalar FMAs the kernel was instruction-bound at a third of the memory bandwidth, and a
// tcgen05 tile (M = 128, TMEM, one issuing thread per CTA) has no use for 4 query rows per token.
// One persistent CTA per SM: a producer warp streams the tasks' K and V tiles (TMA, 128-byte swizzle, so
// that ldmatrix reads them without bank conflicts) through a ring that keeps the whole shared memory in
// flight; twelve consumer warps take the tasks in turn.  (A warp that fetched its own task and then worked on
// it left the memory idle in between: S = 4096, L = 28, 28 heads 325 us.)
// The call has no status word: a task whose bounded wait runs out gets NaN rows.
#include "common.cuh"
#include "sm100.cuh"

namespace sdv {

constexpr int kDh = 128;               // head size
constexpr int kDraftWarps = 12;        // consumer warps
constexpr int kDraftThreads = (kDraftWarps + 1) * 32;
constexpr int kHalf = 32 * 128;        // bytes of one half of a tile: up to 32 layers x 64 values, swizzled
constexpr int kTile = 2 * kHalf;       // K (or V) of one task
// Ring slots are a multiple of the consumer warps (12 for separate K and V, 24 for one buffer; 192 KiB): a slot
// then always belongs to the same warp, which has seen its previous load complete before it waits for the next
// one, so that the parity of the slot's barrier names one phase.  (Fewer slots only where a CTA has no more
// tasks than that and none is used twice.)
constexpr int kMaxRing = 2 * kDraftWarps;
constexpr int kDraftSmem = kMaxRing * kTile;

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// SAME: k and v are one buffer (the un-projected reading); every row is then fetched once and both products
// read the one tile.
template <bool SAME>
__global__ void __launch_bounds__(kDraftThreads, 1)
draft_feature_attention_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                               const uint16_t* qp, long long tasks, int L, int Q, int H, float scale, int stages,
                               int tile_bytes, long long wait_cycles, uint16_t* out) {
    using namespace sm100;
    extern __shared__ uint8_t dsm_raw[];
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int kSlot = SAME ? kTile : 2 * kTile;
    __shared__ __align__(8) uint64_t full[kMaxRing], empty[kMaxRing];
    __shared__ int abort_flag;
    __shared__ __align__(16) uint16_t s_out[kDraftWarps][8 * kDh];                  // a task's output rows, before they leave as whole lines
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        fence_barrier_init();
        prefetch_tensormap(&map_k);
        if (!SAME) prefetch_tensormap(&map_v);
    }
    // rows >= L of every tile stay zero (the copies write L rows)
    for (int t = threadIdx.x; t < stages * (kSlot / kHalf) * (32 - L) * 8; t += kDraftThreads) {
        const int per = (32 - L) * 8, half = t / per, r = t - half * per;
        reinterpret_cast<uint4*>(ring + half * kHalf + L * 128)[r] = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
    __syncthreads();
    begin_dependent(qp, out);
    const int D = H * kDh;
    // this CTA's tasks (token, head), consecutive: their rows are neighbours in memory
    const long long first = tasks * blockIdx.x / gridDim.x;
    const int n = (int)(tasks * (blockIdx.x + 1) / gridDim.x - first);

    if (warp == kDraftWarps) {
        // ---- producer: a whole warp in uniform control flow, one lane elected around the copies
        const uint64_t pol = policy_evict_first();
        int s = (int)(first / H), h = (int)(first - (long long)s * H), slot = 0;
        uint32_t ph = 1;
        for (int i = 0; i < n; ++i) {
            if (!mbar_wait_warp(&empty[slot], ph, &abort_flag, wait_cycles)) { unwind_pause(); break; }
            uint8_t* dst = ring + slot * kSlot;
            if (elect_one()) {
                mbar_arrive_expect_tx(&full[slot], tile_bytes);
                tma_load_3d(dst, &map_k, h * kDh, 0, s, &full[slot], pol);
                tma_load_3d(dst + kHalf, &map_k, h * kDh + 64, 0, s, &full[slot], pol);
                if (!SAME) {
                    tma_load_3d(dst + kTile, &map_v, h * kDh, 0, s, &full[slot], pol);
                    tma_load_3d(dst + kTile + kHalf, &map_v, h * kDh + 64, 0, s, &full[slot], pol);
                }
            }
            __syncwarp();
            if (++h == H) { h = 0; ++s; }
            if (++slot == stages) { slot = 0; ph ^= 1u; }
        }
        return;
    }
    const int g = lane >> 2, t = lane & 3;                                          // mma fragment coordinates
    const int mi = lane >> 3, r = lane & 7;                                         // ldmatrix: matrix and row of this lane
    const float scale_log2 = scale * 1.4426950408889634f;
    int i = warp;
    for (; i < n; i += kDraftWarps) {
        const int s = (int)((first + i) / H), h = (int)(first + i - (long long)s * H);
        const int slot = i % stages;
        const uint32_t ks_addr = smem_u32(ring + slot * kSlot), vs_addr = SAME ? ks_addr : ks_addr + kTile;
        // ---- meta queries of this head as A fragments (row g; rows >= Q and rows 8..15 are zero)
        uint32_t qa[8][2];
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const uint32_t* qr = reinterpret_cast<const uint32_t*>(qp + (size_t)min(g, Q - 1) * D + h * kDh) + t;
            qa[ks][0] = g < Q ? __ldg(qr + ks * 8) : 0u;
            qa[ks][1] = g < Q ? __ldg(qr + ks * 8 + 4) : 0u;
        }
        if (!mbar_wait_warp(&full[slot], (uint32_t)(i / stages) & 1u, &abort_flag, wait_cycles)) break;
        // ---- K rows as B fragments (layer 8 * nt + r; 16-byte piece c of a row sits at piece c ^ (row & 7)) and scores S[q][l]
        float sc[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
            for (int kp = 0; kp < 4; ++kp) {                                        // two k-steps per load
                const int c = 2 * (2 * kp + (mi >> 1)) + (mi & 1);
                uint32_t b0, b1, b2, b3;
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3)
                             : "r"(ks_addr + (c >> 3) * kHalf + (nt * 8 + r) * 128 + (((c & 7) ^ r) << 4)) : "memory");
                mma_bf16_16816(sc[nt], qa[2 * kp][0], 0u, qa[2 * kp][1], 0u, b0, b1);
                mma_bf16_16816(sc[nt], qa[2 * kp + 1][0], 0u, qa[2 * kp + 1][1], 0u, b2, b3);
            }
        }
        // ---- soft-max over the layers: row g lives in the four lanes with this g, columns 8 nt + 2t, + 1
        float mx = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int l0 = nt * 8 + 2 * t;
            sc[nt][0] = l0 < L ? sc[nt][0] * scale_log2 : -INFINITY;
            sc[nt][1] = l0 + 1 < L ? sc[nt][1] * scale_log2 : -INFINITY;
            mx = fmaxf(mx, fmaxf(sc[nt][0], sc[nt][1]));
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        float sum = 0.f;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            sc[nt][0] = exp2f(sc[nt][0] - mx); sc[nt][1] = exp2f(sc[nt][1] - mx);
            sum += sc[nt][0] + sc[nt][1];
        }
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        const float inv = 1.f / sum;
        // probabilities as A fragments of the second product (k = layer): tiles 2 ks and 2 ks + 1
        uint32_t pa[2][2];
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            pa[ks][0] = pack_bf16(sc[2 * ks][0] * inv, sc[2 * ks][1] * inv);
            pa[ks][1] = pack_bf16(sc[2 * ks + 1][0] * inv, sc[2 * ks + 1][1] * inv);
        }
        // ---- out[q][d] = sum_l P[q][l] V[l][d]; V fragments by transposing loads from shared memory
        uint16_t* orow = s_out[warp] + g * kDh + 2 * t;
#pragma unroll
        for (int np = 0; np < 8; ++np) {                                             // 16 output values per step
            float o0[4] = {0.f, 0.f, 0.f, 0.f}, o1[4] = {0.f, 0.f, 0.f, 0.f};
            const int c = 2 * np + (mi >> 1);
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                uint32_t b0, b1, b2, b3;
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3)
                             : "r"(vs_addr + (c >> 3) * kHalf + (ks * 16 + (mi & 1) * 8 + r) * 128 + (((c & 7) ^ r) << 4)) : "memory");
                mma_bf16_16816(o0, pa[ks][0], 0u, pa[ks][1], 0u, b0, b1);
                mma_bf16_16816(o1, pa[ks][0], 0u, pa[ks][1], 0u, b2, b3);
            }
            *reinterpret_cast<uint32_t*>(orow + np * 16) = pack_bf16(o0[0], o0[1]);
            *reinterpret_cast<uint32_t*>(orow + np * 16 + 8) = pack_bf16(o1[0], o1[1]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);                                    // every lane has read the tile
        for (int x = lane; x < Q * 16; x += 32)
            reinterpret_cast<uint4*>(out + ((size_t)s * Q + (x >> 4)) * D + (size_t)h * kDh)[x & 15] =
                reinterpret_cast<const uint4*>(s_out[warp])[x];
        __syncwarp();                                                                // s_out is reused by the next task
    }
    if (i >= n) return;
    for (; i < n; i += kDraftWarps) {                                                // a wait ran out: this warp's rows from there on
        const int s = (int)((first + i) / H), h = (int)(first + i - (long long)s * H);
        for (int x = lane; x < Q * 16; x += 32)
            reinterpret_cast<uint4*>(out + ((size_t)s * Q + (x >> 4)) * D + (size_t)h * kDh)[x & 15] =
                make_uint4(0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu);
    }
    unwind_pause();
}

sd_status launch_draft_feature_attention(const void* qp, const void* k, const void* v, int S, int L, int Q, int H,
                                         float scale, void* out, cudaStream_t st) {
    const int D = H * kDh;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SD_ERR_CUDA;
    const int sms = sm_count(dev);
    const long long tasks = (long long)S * H;
    const bool same = k == v;
    const uint64_t dims[3] = {(uint64_t)D, (uint64_t)L, (uint64_t)S};
    const uint64_t strides[2] = {(uint64_t)D * 2, (uint64_t)L * D * 2};
    const uint32_t box[3] = {64, (uint32_t)L, 1};
    CUtensorMap mk, mv;
    if (!encode_tmap_bf16_3d(&mk, k, dims, strides, box, 128)) return SD_ERR_CUDA;
    if (same) mv = mk;
    else if (!encode_tmap_bf16_3d(&mv, v, dims, strides, box, 128)) return SD_ERR_CUDA;
    const int grid = (int)(tasks < sms ? tasks : sms);
    const int slot = same ? kTile : 2 * kTile;
    int stages = kDraftSmem / slot;                                   // 12 or 24
    const long long most = (tasks + grid - 1) / grid;                 // a CTA's tasks: no more slots than that
    if (stages > most) stages = (int)most;
    const int smem = stages * slot + 1024;
    const TestKnobs knobs = test_knobs();
    auto kern = same ? draft_feature_attention_kernel<true> : draft_feature_attention_kernel<false>;
    if (!allow_dynamic_smem(kern, smem)) return SD_ERR_CUDA;
    const int tile_bytes = (same ? 2 : 4) * L * 128 + (knobs.withhold ? 16 : 0);       // (withheld: bytes that do not come)
    return launch_dependent(kern, dim3(grid), kDraftThreads, smem, 1, st, mk, mv, qp, tasks, L, Q, H, scale, stages, tile_bytes,
                            knobs.wait_cycles, out);
}

}  // namespace sdv
