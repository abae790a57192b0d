// Verification at a sampling temperature of drafts that were SAMPLED from the draft model's distributions q,
// from the logits the LM-head pass kept: trees (sd_accept_tree_sampled_q) and chains
// (sd_accept_chain_sampled with logits).
//
// Every distribution met at a node is max(p - a q, 0) / b with two scalars (a = 0, b = 1 at a node's start; a
// rejection makes a <- a + b, b <- sum_v max(p - a q, 0)), so a rejection costs one reduction over the
// vocabulary.  One cluster of eight CTAs per sequence: every CTA holds its eighth of p (from the logits) and
// q of the current node in REGISTERS (512 threads, entry k * 512 + t of the slice in thread t: coalesced
// loads, all in flight together), adds up its part in a fixed order, and sends the sum to all eight CTAs with
// stores that report to a barrier there; the eight are added in rank order, so all CTAs take the same
// decisions.  The last token is found by inverse CDF in vocabulary order by the CTA whose slice holds the
// crossing.  What bounds it is latency: per node one round of loads, per rejection one exchange.  (With the
// slices in shared memory, 256 threads and two cluster barriers' worth of synchronisation per exchange 8 trees of 60
// nodes took 51 to 65 us at a vocabulary of 152064, now 24 to 25; 8 chains of 10 drafts 31 in four kernels, now 8.  Calls one
// behind another; replayed from a graph, as the figures in draw_token are, 23 to 24 and 6.9.)
#include "tree_device.cuh"
#include "sm100.cuh"

namespace sdv {

constexpr int kQCluster = 8;
constexpr int kQThreads = 512;
constexpr int kQWarps = kQThreads / 32;
// Entries per thread, PER: 40 (V <= 163840), and 16 and 8 where they hold the vocabulary.  The code is unrolled over them, and
// with 40 the way through it is as long however few of them there are.  8 against 40: trees of 60 nodes, 4 sequences, vocabulary
// 4099, the whole tail 38.1 -> 31.6 us, 2 sequences, 32000 68.5 -> 62.3; 16 against 40: 8 sequences, 50257 131.1 -> 127.5.
constexpr int kQPerMax = 40;
constexpr int kQMaxSlice = kQThreads * kQPerMax;       // vocabulary entries per CTA

// mute: test hook, the CTA of a cluster that keeps its sums to itself (-1: none)
struct QWaits { long long cycles; int mute; };

struct QShared {
    uint64_t bar[2];                                   // two exchanges in turn: a CTA may start the next while a peer still
    float cta_sum[2][kQCluster];                       // waits for this one (it cannot get two ahead)
    float warp_sum[kQWarps];
    float run_sum[kQPerMax * kQWarps];                 // the draw: sums of 32 consecutive entries
    float run[kQPerMax][32];                           // the entries of one warp
    int32_t path[kMaxT], par[kMaxT], tok[kMaxT];
    float u[kMaxT], px[kMaxT], qx[kMaxT];
    float acc;
    int abort_flag, bad, pick;
};

__device__ __forceinline__ float warp_sum_f32(float v) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Sums over the warp of N values per lane (N = 8, 16 or 32): lane j, modulo N, gets value j's, added up in the order that
// warp_sum_f32 adds in.  Lanes that hold the same values hand half of them over in each step: 31 and 23 exchanges
// instead of 160 and 40 (a draw's 40 sums took 200).
template <int N>
__device__ __forceinline__ float warp_sums(float* x, int lane) {
#pragma unroll
    for (int d = 16; d >= N; d >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], d);
#pragma unroll
    for (int h = N / 2; h >= 1; h >>= 1)
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = (lane & h) ? x[i + h] : x[i], send = (lane & h) ? x[i] : x[i + h];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    return x[0];
}

// This CTA's part of the vocabulary behind one node
template <int PER>
struct VocabSlice {
    float p[PER], q[PER];
    int len;
    // q: null for a node whose q is not needed
    __device__ __forceinline__ void load(const float* logits, const float* qrow, float inv_temp, float lse, int tid) {
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int i = k * kQThreads + tid;
            p[k] = i < len ? __ldg(logits + i) : -INFINITY;
            q[k] = (qrow && i < len) ? __ldg(qrow + i) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) p[k] = __expf(p[k] * inv_temp - lse);
    }
    __device__ __forceinline__ float at(int k, float a) const { return fmaxf(p[k] - a * q[k], 0.f); }
    __device__ __forceinline__ float thread_sum(float a) const {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < PER; ++k) s[k & 3] += at(k, a);
        return (s[0] + s[1]) + (s[2] + s[3]);
    }
};

// Sum of max(p - a q, 0) over the whole vocabulary, the same bits in every CTA of the cluster; n_red counts the
// exchanges so far.  sh.cta_sum[(n_red - 1) & 1] keeps the eight parts.  false: a peer's part did not arrive.
template <int PER>
__device__ __forceinline__ bool reduce_all(QShared& sh, const VocabSlice<PER>& v, float a, int rank, int tid, const QWaits& waits, int& n_red,
                                           float& all) {
    const int set = n_red & 1;
    const uint32_t phase = (uint32_t)(n_red >> 1) & 1u;
    ++n_red;
    const float w = warp_sum_f32(v.thread_sum(a));
    if ((tid & 31) == 0) sh.warp_sum[tid >> 5] = w;
    __syncthreads();
    if (tid < kQCluster) {
        float total = 0.f;
#pragma unroll
        for (int i = 0; i < kQWarps; ++i) total += sh.warp_sum[i];
        if (tid == rank) {
            sh.cta_sum[set][rank] = total;
            sm100::mbar_arrive_expect_tx(&sh.bar[set], (kQCluster - 1) * 4);
        } else if (rank != waits.mute) {
            sm100::st_async_b32(sm100::map_dsmem(sm100::smem_u32(&sh.cta_sum[set][rank]), (uint32_t)tid), __float_as_uint(total),
                                sm100::map_dsmem(sm100::smem_u32(&sh.bar[set]), (uint32_t)tid));
        }
    }
    const bool ok = sm100::mbar_wait_cluster(&sh.bar[set], phase, &sh.abort_flag, waits.cycles);
    __syncthreads();                                   // (warp_sum may be written again; the abort flag is everybody's)
    all = 0.f;
#pragma unroll
    for (int r = 0; r < kQCluster; ++r) all += sh.cta_sum[set][r];
    return ok && *reinterpret_cast<volatile int*>(&sh.abort_flag) == 0;
}

// The token at which the cumulative mass of max(p - a q, 0), in vocabulary order, reaches w * (total mass); the
// latest exchange summed exactly this distribution.  Every CTA calls it, the owner of the crossing writes.
template <int PER>
__device__ __forceinline__ void draw_token(QShared& sh, const VocabSlice<PER>& v, float a, float w, float total, int n_red, int rank,
                                           int tid, int v0, int32_t* out_slot, int32_t* status) {
    const float* parts = sh.cta_sum[(n_red - 1) & 1];
    const int warp = tid >> 5, lane = tid & 31;
    const float target = w * total;
    float before = 0.f;
    int owner = -1, last_with_mass = -1;
    for (int r = 0; r < kQCluster; ++r) {
        const float x = parts[r];
        if (x > 0.f) last_with_mass = r;
        if (owner < 0 && x > 0.f && before + x >= target) owner = r;
        if (owner < 0) before += x;
    }
    if (owner < 0) {                                   // rounding left the sum short: the last slice with mass
        owner = last_with_mass;
        if (owner >= 0) before -= parts[owner];
    }
    if (owner < 0) {                                   // no mass at all (inputs not finite, or vanished by rounding)
        if (rank == 0 && tid == 0) { set_status(status, SD_ERR_BOUNDS); *out_slot = 0; }
        return;
    }
    if (rank != owner) return;
    // which 32 consecutive entries, then which of them
    const int rows = (v.len + kQThreads - 1) / kQThreads;
    {
        float x[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) x[k] = v.at(k, a);
        constexpr int kFirst = PER > 32 ? 32 : PER;
        static_assert(kFirst == PER || PER == 40, "32 rows and 8");
        const float s = warp_sums<kFirst>(x, lane);
        if (lane < kFirst) sh.run_sum[lane * kQWarps + warp] = s;
        if constexpr (PER > 32) {
            const float s8 = warp_sums<8>(x + 32, lane);
            if (lane < 8) sh.run_sum[(32 + lane) * kQWarps + warp] = s8;
        }
    }
    __syncthreads();
    if (warp == 0) {
        float acc = before;
        int lastp = -1;
        int t = warp_find_crossing(sh.run_sum, rows * kQWarps, target, &acc, &lastp, lane);
        if (t < 0) { t = max(lastp, 0); acc -= sh.run_sum[t]; }
        if (lane == 0) { sh.acc = acc; sh.pick = t; }
    }
    __syncthreads();
    const int t = sh.pick;
    if (warp == (t & (kQWarps - 1))) {
        // All rows, not only the one looked for: with 8 and 16 entries the compiler took a selected one for an indexed array,
        // which put the slice into local memory (per call, 8 sequences of 60 nodes: V 32000 8.9 -> 8.0 us, 50257 10.5 -> 8.8,
        // chains of 11 5.7 -> 4.7 and 6.8 -> 5.5; with 40, 152064, 16.3 -> 16.2 and 7.4 -> 6.8).
#pragma unroll
        for (int k = 0; k < PER; ++k) sh.run[k][lane] = v.at(k, a);
        __syncwarp();
        float acc = sh.acc;
        int lastp = -1;
        int e = warp_find_crossing(sh.run[t / kQWarps], 32, target, &acc, &lastp, lane);
        if (e < 0) e = max(lastp, 0);
        if (lane == 0) *out_slot = v0 + t * 32 + e;
    }
}

// Set-up shared by the two kernels: barriers, and this cluster's CTAs know of each other's.
__device__ __forceinline__ void q_begin(QShared& sh, int tid) {
    if (tid == 0) {
        sh.abort_flag = 0;
        sh.bad = 0;
        sm100::mbar_init(&sh.bar[0], 1);
        sm100::mbar_init(&sh.bar[1], 1);
        sm100::fence_barrier_init();
    }
    sm100::cluster_arrive_release();
    sm100::cluster_wait_acquire();
}
// nobody leaves while a peer may still send to it, or has sent what was not waited for
__device__ __forceinline__ void q_end(QShared& sh) {
    __syncwarp();
    sm100::cluster_arrive_relaxed();
    sm100::cluster_wait_acquire();
    if (*reinterpret_cast<volatile int*>(&sh.abort_flag)) sm100::unwind_pause();
}

template <int PER>
__global__ void __launch_bounds__(kQThreads, 1)
tree_walk_q_kernel(sd_batch bt, int V, float inv_temp, const float* lse, const float* logits, const int32_t* draft,
                   const float* q_rows, const float* u, const float* w, int32_t* n_acc, int32_t* path, int32_t* out_tok,
                   int32_t* new_len, int32_t* status, const QWaits waits) {
    __shared__ QShared sh;
    const int tid = threadIdx.x, lane = tid & 31;
    q_begin(sh, tid);
    begin_dependent(bt, lse, logits, draft, q_rows, u, w);
    const int b = blockIdx.x / kQCluster;
    const int rank = (int)sm100::cluster_ctarank();
    const int T = bt.T_max;
    const int slice = (V + kQCluster - 1) / kQCluster;
    const int v0 = min(V, rank * slice);
    VocabSlice<PER> v;
    v.len = min(V, v0 + slice) - v0;
    const int n = bt.n_nodes[b];
    // the tree, checked by every CTA in the same way
    const bool n_ok = n >= 1 && n <= T;
    if (tid < T) {                                     // (unused nodes too: the loads need not wait for n)
        const size_t at = (size_t)b * T + tid;
        const int p = bt.parents[at], x = draft[at];
        sh.par[tid] = p; sh.tok[tid] = x; sh.u[tid] = u[at];
        if (!n_ok || tid >= n) {}
        else if (tid == 0 ? (p != -1) : (p < 0 || p >= tid)) sh.bad = SD_ERR_INVALID_TREE;
        else if (tid > 0 && (x < 0 || x >= V)) atomicCAS(&sh.bad, 0, (int)SD_ERR_BOUNDS);
    }
    __syncthreads();
    const int bad = n_ok ? sh.bad : (int)SD_ERR_INVALID_TREE;
    if (bad != 0) {                                    // (the same in every CTA)
        if (rank == 0 && tid == 0) { set_status(status, bad); n_acc[b] = 0; }
        q_end(sh);
        return;
    }
    const int par0 = lane < n ? sh.par[lane] : -2, par1 = lane + 32 < n ? sh.par[lane + 32] : -2;
    int cur = 0, na = 1, n_red = 0;
    float a = 0.f, bsum = 1.f;
    bool ok = true;
    if (tid == 0) sh.path[0] = 0;
    while (ok) {
        const size_t row = (size_t)b * T + cur;
        const float row_lse = lse[row];
        const float* lrow = logits + row * V;
        const float* qrow = q_rows + row * V;
        v.load(lrow + v0, qrow + v0, inv_temp, row_lse, tid);
        if (tid < n && sh.par[tid] == cur) {           // p and q of the children's tokens, together with the slices
            sh.px[tid] = __expf(__ldg(lrow + sh.tok[tid]) * inv_temp - row_lse);
            sh.qx[tid] = __ldg(qrow + sh.tok[tid]);
        }
        uint64_t kids = ((uint64_t)__ballot_sync(0xffffffffu, par1 == cur) << 32) | __ballot_sync(0xffffffffu, par0 == cur);
        __syncthreads();
        a = 0.f; bsum = 1.f;
        int nxt = -1;
        bool summed = false;                           // the latest exchange summed this node's distribution
        while (kids) {                                 // children of cur in node order (the same walk in every thread)
            const int c = __ffsll((long long)kids) - 1;
            kids &= kids - 1;
            if (sh.u[c] * bsum * sh.qx[c] < fmaxf(sh.px[c] - a * sh.qx[c], 0.f)) { nxt = c; break; }
            a += bsum;
            ok = reduce_all(sh, v, a, rank, tid, waits, n_red, bsum);
            summed = true;
            if (!ok) break;
        }
        if (!ok) break;
        if (nxt < 0) {
            if (!summed) ok = reduce_all(sh, v, a, rank, tid, waits, n_red, bsum);   // nothing rejected here: all of p
            break;
        }
        if (tid == 0) sh.path[na] = nxt;
        cur = nxt;
        ++na;
    }
    __syncthreads();
    if (!ok) {
        if (tid == 0) set_status(status, SD_ERR_TIMEOUT);
    } else {
        if (rank == 0) {
            for (int k = tid; k < T; k += kQThreads) {
                path[(size_t)b * T + k] = k < na ? sh.path[k] : -1;
                if (k != na - 1) out_tok[(size_t)b * T + k] = k + 1 < na ? sh.tok[sh.path[k + 1]] : -1;
            }
            if (tid == 0) { n_acc[b] = na; new_len[b] = bt.len[b] + na; }
        }
        draw_token(sh, v, a, w[b], bsum, n_red, rank, tid, v0, out_tok + (size_t)b * T + na - 1, status);
    }
    q_end(sh);
}

// Chains: node j's token is kept iff u * q(token) < p(token), p and q behind node j - 1; the walk stops at the
// first rejection, and the last token comes from max(p - q, 0) there, or from p of the leaf.  Only the stop
// node's row of p and q is needed, so the whole rule is one kernel with one exchange.
template <int PER>
__global__ void __launch_bounds__(kQThreads, 1)
chain_walk_q_logits_kernel(sd_batch bt, int V, float inv_temp, const float* lse, const float* logits, const int32_t* draft,
                           const float* q_tok, const float* q_rows, const float* u, const float* w, int32_t* n_acc, int32_t* path,
                           int32_t* out_tok, int32_t* new_len, int32_t* status, const QWaits waits) {
    __shared__ QShared sh;
    __shared__ uint32_t s_rejected[2];
    const int tid = threadIdx.x;
    q_begin(sh, tid);
    begin_dependent(bt, lse, logits, draft, q_tok, q_rows, u, w);
    const int b = blockIdx.x / kQCluster;
    const int rank = (int)sm100::cluster_ctarank();
    const int T = bt.T_max;
    const int slice = (V + kQCluster - 1) / kQCluster;
    const int v0 = min(V, rank * slice);
    VocabSlice<PER> v;
    v.len = min(V, v0 + slice) - v0;
    const int n = bt.n_nodes[b];
    const bool n_ok = n >= 1 && n <= T;
    if (tid < 64) {
        bool rejected = false;
        if (tid < T) {                                 // (unused nodes too: the loads need not wait for n)
            const size_t at = (size_t)b * T + tid;
            const int p = bt.parents[at], x = draft[at];
            const float uq = u[at], qt = q_tok[at], plse = tid > 0 ? lse[at - 1] : 0.f;
            const bool x_ok = x >= 0 && x < V;
            const float px = tid > 0 && x_ok ? __expf(__ldg(logits + (at - 1) * V + x) * inv_temp - plse) : 0.f;
            sh.tok[tid] = x;
            if (n_ok && tid < n) {
                if (tid == 0 ? (p != -1) : (p < 0 || p >= tid)) sh.bad = SD_ERR_INVALID_TREE;
                else if (tid > 0 && p != tid - 1) atomicCAS(&sh.bad, 0, (int)SD_ERR_UNSUPPORTED);      // the tree branches
                if (tid > 0 && !x_ok) set_status(status, SD_ERR_BOUNDS);
                rejected = tid > 0 && !(uq * qt < px);
            }
        }
        const uint32_t m = __ballot_sync(0xffffffffu, rejected);
        if ((tid & 31) == 0) s_rejected[tid >> 5] = m;
    }
    __syncthreads();
    const int bad = n_ok ? sh.bad : (int)SD_ERR_INVALID_TREE;
    if (bad != 0) {                                    // (the same in every CTA)
        if (rank == 0 && tid == 0) { set_status(status, bad); n_acc[b] = 0; }
        q_end(sh);
        return;
    }
    const uint32_t lo = s_rejected[0], hi = s_rejected[1];
    const int na = lo ? __ffs(lo) - 1 : (hi ? 32 + __ffs(hi) - 1 : n);       // the first rejected node, or all
    const size_t row = (size_t)b * T + na - 1;
    const float a = na < n ? 1.f : 0.f;
    v.load(logits + row * V + v0, na < n ? q_rows + row * V + v0 : nullptr, inv_temp, lse[row], tid);
    if (rank == 0) {
        for (int k = tid; k < T; k += kQThreads) {
            path[(size_t)b * T + k] = k < na ? k : -1;
            if (k != na - 1) out_tok[(size_t)b * T + k] = k + 1 < na ? sh.tok[k + 1] : -1;
        }
        if (tid == 0) { n_acc[b] = na; new_len[b] = bt.len[b] + na; }
    }
    int n_red = 0;
    float total = 0.f;
    if (reduce_all(sh, v, a, rank, tid, waits, n_red, total))
        draw_token(sh, v, a, w[b], total, n_red, rank, tid, v0, out_tok + (size_t)b * T + na - 1, status);
    else if (tid == 0)
        set_status(status, SD_ERR_TIMEOUT);
    q_end(sh);
}

static QWaits q_waits() {
    const TestKnobs knobs = test_knobs();
    return {knobs.wait_cycles, knobs.withhold ? 1 : -1};
}

bool q_kernels_hold(int V) { return (V + kQCluster - 1) / kQCluster <= kQMaxSlice; }

sd_status launch_accept_tree_sampled_q(const sd_batch& bt, int V, float inv_temp, const float* lse, const float* logits,
                                       const int32_t* draft, const float* q_rows, const float* u, const float* w,
                                       int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len,
                                       int32_t* dev_status, cudaStream_t st) {
    if (!q_kernels_hold(V)) return SD_ERR_UNSUPPORTED;
    const int slice = (V + kQCluster - 1) / kQCluster;
    auto kern = slice <= 8 * kQThreads ? tree_walk_q_kernel<8> : (slice <= 16 * kQThreads ? tree_walk_q_kernel<16> : tree_walk_q_kernel<kQPerMax>);
    return launch_dependent(kern, dim3(bt.B * kQCluster), kQThreads, 0, kQCluster, st, bt, V, inv_temp, lse, logits, draft,
                            q_rows, u, w, n_acc, path, out_tok, new_len, dev_status, q_waits());
}

sd_status launch_accept_chain_logits(const sd_batch& bt, int V, float inv_temp, const float* lse, const float* logits,
                                     const int32_t* draft, const float* q_tok, const float* q_rows, const float* u, const float* w,
                                     int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len, int32_t* dev_status,
                                     cudaStream_t st) {
    const int slice = (V + kQCluster - 1) / kQCluster;
    auto kern = slice <= 8 * kQThreads ? chain_walk_q_logits_kernel<8>
                                       : (slice <= 16 * kQThreads ? chain_walk_q_logits_kernel<16> : chain_walk_q_logits_kernel<kQPerMax>);
    return launch_dependent(kern, dim3(bt.B * kQCluster), kQThreads, 0, kQCluster, st, bt, V, inv_temp, lse, logits,
                            draft, q_tok, q_rows, u, w, n_acc, path, out_tok, new_len, dev_status, q_waits());
}

}  // namespace sdv
