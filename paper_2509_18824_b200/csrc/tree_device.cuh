// Device-side pieces shared by the stand-alone kernels (acceptance, compaction, LM-head merge) and
// the fused tail kernel that runs the three back to back for one sequence per CTA.
#pragma once
#include "common.cuh"

namespace sdv {

constexpr int kLayersPerLaunch = 64;     // layer descriptors travel as kernel parameters
constexpr int kLmMaxCols = 512;          // hidden rows per LM-head pass = row stride of the candidate tables

struct CompactLayers {
    uint4* kc[kLayersPerLaunch];
    uint4* vc[kLayersPerLaunch];
    const uint4* kt[kLayersPerLaunch];
    const uint4* vt[kLayersPerLaunch];
    int32_t num_blocks[kLayersPerLaunch];
};

// descriptors of layers [l0, l0 + nl) (implemented beside the compaction kernel)
void fill_compact_layers(CompactLayers* ly, const sd_kv_layer* layers, const void* const* kt, const void* const* vt,
                         int l0, int nl);

__device__ __forceinline__ float key_to_float(int32_t k) {
    return __int_as_float(k < 0 ? (k ^ 0x7fffffff) : k);
}

// (key, index) candidates: larger key wins, lower index among equal keys
__device__ __forceinline__ void take_better(int32_t& k, int32_t& i, int32_t k2, int32_t i2) {
    if (k2 > k || (k2 == k && i2 < i)) { k = k2; i = i2; }
}

__device__ __forceinline__ float ex2_lm(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// running (reference, sum) of a row's soft-max statistics takes in a new partial (ref2, sum2):
// sum counts 2^((logit - ref) * c2)
__device__ __forceinline__ void merge_sumexp(float& ref, float& sum, float ref2, float sum2, float c2) {
    if (!(sum2 > 0.f)) return;
    if (ref2 > ref) { sum = sum * ex2_lm((ref - ref2) * c2) + sum2; ref = ref2; }
    else            { sum += sum2 * ex2_lm((ref2 - ref) * c2); }
}

// Arg-max candidates of up to 64 hidden rows (columns col0 .. + rows - 1), merged by a CTA of 512 threads: lanes along the
// columns, so that a load touches one or two lines of a table, an eighth of the CTAs' candidates per two warps (all eight threads of a row
// in one warp, eight lines per load: 3.1 us of the tail kernel, now 1.8).  Threads 0 .. rows - 1 return row threadIdx.x's.
struct ArgmaxShared { int32_t key[8][64], idx[8][64]; };
__device__ __forceinline__ void merge_rows_argmax(ArgmaxShared& sh, const int32_t* part_key, const int32_t* part_idx, int n_ctas,
                                                  int row_stride, int col0, int rows, int32_t& k, int32_t& i) {
    k = INT32_MIN; i = 0x7fffffff;
    if (n_ctas <= 8) {                                     // one candidate per lane: eight lanes to a row after all
        const int row = threadIdx.x >> 3, c = threadIdx.x & 7;
        if (row < rows && c < n_ctas) {
            k = part_key[(size_t)c * row_stride + col0 + row];
            i = part_idx[(size_t)c * row_stride + col0 + row];
        }
#pragma unroll
        for (int d = 1; d <= 4; d <<= 1) {
            const int32_t k2 = __shfl_xor_sync(0xffffffffu, k, d), i2 = __shfl_xor_sync(0xffffffffu, i, d);
            take_better(k, i, k2, i2);
        }
        if (c == 0) { sh.key[0][row] = k; sh.idx[0][row] = i; }
        __syncthreads();
        k = sh.key[0][threadIdx.x & 63]; i = sh.idx[0][threadIdx.x & 63];
        return;
    }
    const int row = threadIdx.x & 63, part = threadIdx.x >> 6;
    if (row < rows) {
        // (the loads of a batch are issued together: one memory latency instead of a chain of them)
        constexpr int kAhead = 20;                         // 148 CTAs: 19 per thread
        for (int c0 = part; c0 < n_ctas; c0 += 8 * kAhead) {
            int32_t pk[kAhead], pi[kAhead];
#pragma unroll
            for (int a = 0; a < kAhead; ++a) {
                const int c = c0 + 8 * a;
                if (c < n_ctas) {
                    pk[a] = part_key[(size_t)c * row_stride + col0 + row];
                    pi[a] = part_idx[(size_t)c * row_stride + col0 + row];
                }
            }
#pragma unroll
            for (int a = 0; a < kAhead; ++a)
                if (c0 + 8 * a < n_ctas) take_better(k, i, pk[a], pi[a]);
        }
    }
    sh.key[part][row] = k; sh.idx[part][row] = i;
    __syncthreads();
    if ((int)threadIdx.x < rows)
        for (int w = 1; w < 8; ++w) take_better(k, i, sh.key[w][row], sh.idx[w][row]);
}

// Candidates and soft-max partials of eight hidden rows (columns col0 .. + 7 of the per-CTA tables; those from col_end on
// are not read), merged by a CTA of 256 threads.  Lanes 0 .. 7 of a warp, 8 .. 15, ... read one table row each, so that
// a load touches four lines of the tables and not 32; all loads of a thread are in flight together; the sums are
// brought to the largest reference of the row and added up in a fixed order.  Warp w returns row w's log sum
// exp(logit / temperature) (natural log) and arg-max candidate (key, index) in all lanes.  Every thread must call this.
// (Latency and the load path are what it takes: with eight lanes per row, 19 partials one after the other in each, the
// sampled tail of 480 rows spent 4.4 us here, and the merge kernel took 6.5; see sampled_tail_kernel.)
constexpr int kLmMaxCtas = 256;          // CTAs of an LM-head pass
struct MergeShared { float ref[8][8], sum[8][8]; int32_t key[8][8], idx[8][8]; };      // [warp][row]
__device__ __forceinline__ float merge_rows_stats(MergeShared& sh, const int32_t* __restrict__ part_key, const int32_t* __restrict__ part_idx,
                                                  const float* __restrict__ part_ref, const float* __restrict__ part_sum,
                                                  int n_ctas, int row_stride, int col0, int col_end, float c2, int32_t& k, int32_t& i) {
    constexpr int kPer = kLmMaxCtas / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, col = col0 + (lane & 7);
    // one row's (reference, sum) from several: those without mass, or that are no numbers, do not count
    auto rescaled = [&](float r, float sum, float ref) { return !(sum > 0.f) ? 0.f : (r == ref ? sum : sum * ex2_lm((r - ref) * c2)); };
    int32_t pk[kPer], pi[kPer];
    float pr[kPer], ps[kPer];
#pragma unroll
    for (int a = 0; a < kPer; ++a) {
        const int c = warp * 4 + (lane >> 3) + 32 * a;
        pk[a] = INT32_MIN; pi[a] = 0x7fffffff; pr[a] = -INFINITY; ps[a] = 0.f;
        if (c < n_ctas && col < col_end) {
            const size_t at = (size_t)c * row_stride + col;
            pk[a] = __ldcg(part_key + at); pi[a] = __ldcg(part_idx + at);
            pr[a] = __ldcg(part_ref + at); ps[a] = __ldcg(part_sum + at);
        }
    }
    k = INT32_MIN; i = 0x7fffffff;
    float rf = -INFINITY, sm = 0.f;
#pragma unroll
    for (int a = 0; a < kPer; ++a) {
        take_better(k, i, pk[a], pi[a]);
        if (ps[a] > 0.f) rf = fmaxf(rf, pr[a]);
    }
#pragma unroll
    for (int d = 8; d <= 16; d <<= 1) rf = fmaxf(rf, __shfl_xor_sync(0xffffffffu, rf, d));
#pragma unroll
    for (int a = 0; a < kPer; ++a) sm += rescaled(pr[a], ps[a], rf);
    auto across = [&](int d) {
        const int32_t k2 = __shfl_xor_sync(0xffffffffu, k, d), i2 = __shfl_xor_sync(0xffffffffu, i, d);
        take_better(k, i, k2, i2);
        sm += __shfl_xor_sync(0xffffffffu, sm, d);
    };
    across(8); across(16);
    if (lane < 8) { sh.ref[warp][lane] = rf; sh.sum[warp][lane] = sm; sh.key[warp][lane] = k; sh.idx[warp][lane] = i; }
    __syncthreads();
    const int w = lane & 7;                                // this warp's row, warp w's share of it
    rf = sh.ref[w][warp]; sm = sh.sum[w][warp]; k = sh.key[w][warp]; i = sh.idx[w][warp];
    float top = sm > 0.f ? rf : -INFINITY;
#pragma unroll
    for (int d = 1; d <= 4; d <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
    sm = rescaled(rf, sm, top);
    across(1); across(2); across(4);
    return (top * c2 + log2f(sm)) * 0.6931471805599453f;
}

// Where the running sum *acc_io + v[0] + v[1] + ... first reaches `target`, among the elements with
// v > 0 (all v >= 0), found by one warp in a few rounds: the range is cut into 32 consecutive pieces,
// every lane sums one, an inclusive scan over the lanes gives each piece's end value, and the search
// goes on inside the first piece that has mass and whose end value reaches the target, until the
// pieces are single elements.  Every addition happens in a fixed order, so the answer is the same in
// every run.  Returns the index, or -1 when the whole sum stays short; *acc_io then holds the running
// sum in front of the returned element (all of it for -1); *last_pos the last index with v > 0, if any.
// One level down the same elements are added in smaller pieces: where that leaves the refined search
// a rounding short of the target, the piece's last element with mass is the answer.
__device__ __forceinline__ int warp_find_crossing(const float* v, int n, float target, float* acc_io, int* last_pos, int lane) {
    int lo = 0, hi = n;
    float base = *acc_io;
    for (bool top = true;; top = false) {
        const int chunk = (hi - lo + 31) / 32;
        const int i0 = min(hi, lo + lane * chunk), i1 = min(hi, i0 + chunk);
        float sum = 0.f;
        int lastp = -1;
        for (int i = i0; i < i1; ++i) {
            const float x = v[i];
            sum += x;
            if (x > 0.f) lastp = i;
        }
        float incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        float excl = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) excl = 0.f;
        const int lp = __reduce_max_sync(0xffffffffu, lastp);
        if (top && last_pos && lp >= 0) *last_pos = lp;
        const uint32_t cand = __ballot_sync(0xffffffffu, sum > 0.f && base + incl >= target);
        if (!cand) {
            const float all = base + __shfl_sync(0xffffffffu, incl, 31);
            if (top) { *acc_io = all; return -1; }
            *acc_io = all - v[lp];                                   // (lp >= 0: the piece was chosen for having mass)
            return lp;
        }
        const int L0 = __ffs(cand) - 1;
        base += __shfl_sync(0xffffffffu, excl, L0);
        lo = __shfl_sync(0xffffffffu, i0, L0);
        hi = __shfl_sync(0xffffffffu, i1, L0);
        if (chunk == 1) { *acc_io = base; return lo; }
    }
}

// Greedy acceptance for one sequence of n nodes and len cached tokens, executed by one warp.  par/dt/tg: the
// sequence's parents, draft tokens and target arg-max, in global or shared memory (in the tail kernel, where they can be
// brought there meanwhile, 2.9 -> 2.4 us; the stand-alone kernel, which would wait for them, takes 3.6 instead of 4.0 without).  Returns the number of
// accepted nodes (0 for a bad tree, which is reported through *status) and, in lane 0, has written
// n_acc, new_len, path and out_tok; `path_out` (nullable, e.g. shared memory) receives the path too.
__device__ __forceinline__ int accept_sequence(int T, int b, int lane, int n, int len, const int32_t* par,
                                               const int32_t* dt, const int32_t* tg,
                                               int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len,
                                               int32_t* path_out, int32_t* status) {
    bool bad = (n < 1 || n > T);
    if (!bad)
        for (int i = lane; i < n; i += 32) {
            int p = par[i];
            if (i == 0 ? (p != -1) : (p < 0 || p >= i)) bad = true;
        }
    if (__any_sync(0xffffffffu, bad)) {
        if (lane == 0) set_status(status, SD_ERR_INVALID_TREE);
        return 0;
    }
    // key = depth * 64 + (63 - index) for valid nodes: max key = deepest, lowest index.  A lane walks up from its
    // two nodes at the same time.
    int j0 = lane < n ? lane : 0, j1 = lane + 32 < n ? lane + 32 : 0;
    int d0 = 0, d1 = 0;
    bool ok0 = lane < n, ok1 = lane + 32 < n;
    for (int step = 0; step < kMaxT && (j0 > 0 || j1 > 0); ++step) {
        if (j0 > 0) { const int p = par[j0]; ok0 = ok0 && dt[j0] == tg[p]; ++d0; j0 = p; }
        if (j1 > 0) { const int p = par[j1]; ok1 = ok1 && dt[j1] == tg[p]; ++d1; j1 = p; }
    }
    int best_key = ok0 ? d0 * 64 + (63 - lane) : -1;
    if (ok1) best_key = max(best_key, d1 * 64 + (31 - lane));
    best_key = __reduce_max_sync(0xffffffffu, best_key);   // node 0 is always valid
    const int best = 63 - (best_key & 63);
    const int na = (best_key >> 6) + 1;
    int32_t* pa = path + (size_t)b * T;
    int32_t* ot = out_tok + (size_t)b * T;
    for (int k = na + lane; k < T; k += 32) { pa[k] = -1; ot[k] = -1; }
    if (lane == 0) {
        n_acc[b] = na;
        new_len[b] = len + na;
        int j = best;
        for (int k = na - 1; k >= 0; --k) {
            pa[k] = j;
            if (path_out) path_out[k] = j;
            if (k >= 1) ot[k - 1] = dt[j];
            j = par[j];
        }
        ot[na - 1] = tg[best];
    }
    return na;
}

// Copies the accepted rows of sequence b in layers [l0, l0 + n_layers): work items idx = tid, tid + stride, ...
// One item = one 16-byte vector of one (layer, accepted node, K or V, KV head).  `path` holds the
// sequence's accepted nodes (global or shared memory).
template <int kLayers = 1>
__device__ __forceinline__ void compact_sequence(const sd_batch& bt, const CompactLayers& ly, int l0, int n_layers, int b,
                                                 int na, const int32_t* path, int tid, int stride,
                                                 int32_t* status) {
    const int T = bt.T_max;
    const int len = bt.len[b];
    const int vec_per_head = bt.D * 2 / 16;               // 16 for D = 128
    const int vec_per_node = bt.Hkv * vec_per_head;       // per K or V
    const int per_layer = na * 2 * vec_per_node;
    const int total = per_layer * n_layers;
    const int per_node = 2 * vec_per_node;                 // K and V vectors of one node
    if (stride % per_node == 0) {
        // Every thread keeps its place inside a node (K or V, head, 16-byte piece) and only walks over
        // the accepted nodes and the layers: no index arithmetic beyond the two table look-ups per vector.
        const int sub = tid % per_node;
        const int is_v = sub / vec_per_node;
        const int kvh = (sub - is_v * vec_per_node) / vec_per_head;
        const int c = sub - is_v * vec_per_node - kvh * vec_per_head;
        const int k_step = stride / per_node;
        constexpr int kUnroll = 4;                         // nodes in flight per thread: loads before stores
        for (int k0 = tid / per_node; k0 < na; k0 += k_step * kUnroll) {
            size_t src[kUnroll], dst[kUnroll];
            int blk[kUnroll];
            bool has[kUnroll];                             // this slot holds an accepted node
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int k = k0 + u * k_step;
                blk[u] = -1;
                has[u] = false;
                if (k >= na) continue;
                const int node = path[k];
                const int t = len + k;
                if (node < 0 || node >= T || t < 0 || t / kBlock >= bt.max_blocks_per_seq) {
                    set_status(status, SD_ERR_BOUNDS);
                    continue;
                }
                has[u] = true;
                blk[u] = bt.block_table[(size_t)b * bt.max_blocks_per_seq + t / kBlock];
                src[u] = (((size_t)b * T + node) * bt.Hkv + kvh) * vec_per_head + c;
                dst[u] = (((size_t)(blk[u] < 0 ? 0 : blk[u]) * bt.Hkv + kvh) * kBlock + (t % kBlock)) * vec_per_head + c;
            }
            // (kLayers at a time, loaded together before any is stored.  A CTA with several layers: two at a time, four layers
            // of five rows 4.7 -> 3 us; with one layer the longer code only takes longer to fetch, 1.4 -> 1.9 us.)
            for (int l = l0; l < l0 + n_layers; l += kLayers) {
                const uint4* from[kLayers];
                uint4* to[kLayers];
                int nb[kLayers];
#pragma unroll
                for (int i = 0; i < kLayers; ++i) {
                    const int at = kLayers == 1 ? l : min(l + i, l0 + n_layers - 1);
                    from[i] = is_v ? ly.vt[at] : ly.kt[at];
                    to[i] = is_v ? ly.vc[at] : ly.kc[at];
                    nb[i] = ly.num_blocks[at];
                }
                uint4 val[kLayers][kUnroll];
                bool live[kLayers][kUnroll];
#pragma unroll
                for (int i = 0; i < kLayers; ++i)
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        const bool due = has[u] && (kLayers == 1 || l + i < l0 + n_layers);
                        live[i][u] = due && blk[u] >= 0 && blk[u] < nb[i];
                        if (due && !live[i][u]) set_status(status, SD_ERR_BOUNDS);
                        if (live[i][u]) val[i][u] = from[i][src[u]];
                    }
#pragma unroll
                for (int i = 0; i < kLayers; ++i)
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u)
                        if (live[i][u]) to[i][dst[u]] = val[i][u];
            }
        }
        return;
    }
    for (int idx = tid; idx < total; idx += stride) {
        const int li = idx / per_layer;
        const int l = l0 + li;
        int rem = idx - li * per_layer;
        const int k = rem / (2 * vec_per_node);
        rem -= k * 2 * vec_per_node;
        const int is_v = rem / vec_per_node;
        rem -= is_v * vec_per_node;
        const int kvh = rem / vec_per_head;
        const int c = rem - kvh * vec_per_head;
        const int node = path[k];
        const int t = len + k;
        if (node < 0 || node >= T || t < 0 || t / kBlock >= bt.max_blocks_per_seq) {
            set_status(status, SD_ERR_BOUNDS);
            continue;
        }
        const int blk = bt.block_table[(size_t)b * bt.max_blocks_per_seq + t / kBlock];
        if (blk < 0 || blk >= ly.num_blocks[l]) {
            set_status(status, SD_ERR_BOUNDS);
            continue;
        }
        const size_t src = (((size_t)b * T + node) * bt.Hkv + kvh) * vec_per_head + c;
        const size_t dst = (((size_t)blk * bt.Hkv + kvh) * kBlock + (t % kBlock)) * vec_per_head + c;
        if (is_v) ly.vc[l][dst] = ly.vt[l][src];
        else      ly.kc[l][dst] = ly.kt[l][src];
    }
}

}  // namespace sdv
