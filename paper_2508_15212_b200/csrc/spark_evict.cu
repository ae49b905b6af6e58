// Token eviction pre-step of spark_compress (token_budget > 0).
//
// The paper applies channel pruning on top of a token-eviction method and only cites that method's
// settings (App. "Implementation": observation window 32, max-pool kernel 7).  The rule implemented here
// is the benchmark's: for every KV head, the window queries of its G query heads attend (causally inside
// the window) to all earlier keys; the softmax probabilities of the prefix tokens are summed over the
// G*W query rows ("votes"), max-pooled over `pool` neighbours, and the (budget - W) prefix tokens with
// the largest pooled vote (ties: lower position) are kept together with the W window tokens, in
// original order.  Sequences no longer than the budget are kept whole.
//
// Kernels (fp32 CUDA-core arithmetic; this step is preparation, not the timed decode step):
//   evict_scores_kernel<pass 1>  per 128-token tile and query row: max and sum of exp of the scores
//   evict_rowstats_kernel        merge the tile partials into the row's softmax normaliser
//   evict_scores_kernel<pass 2>  recompute the tile's scores, accumulate the column sums = votes
//   evict_select_kernel          pooled max of the votes, exact radix select of the k-th largest, ordered compaction
//                                of the kept positions into kept_tokens: one launch, a cluster per unit; with up to 256 units
//                                (norm_in_select) also the window norm
// Column sums are accumulated inside one CTA in a fixed order, so the votes are reproducible.
#include <cooperative_groups.h>

#include <type_traits>

#include "spark_common.cuh"

namespace spark {

constexpr int kEvTile = 128;          // tokens per CTA tile
constexpr int kEvRows = 64;           // query rows per pass over the tile
constexpr int kEvThreads = 256;
constexpr int kEvStride = kHeadDim + 1;   // padded row length in shared memory (floats)

struct EvictArgs {
    const void* q_win;
    const void* k;
    int64_t sb, sh, st;
    const int32_t* seq_lens;
    int Hq, Hkv, W, budget, pool;
    int S_max, n_tiles;
    float* partial;      // [units][R][n_tiles][2]
    float* rowstat;      // [units][R][2]
    float* votes;        // [units][S_max]
    unsigned* pooled;    // [units][S_max] pooled votes as order-preserving keys (shares above key_cap only)
    int key_cap;         // keys a CTA of the select kernel holds in shared memory
    int32_t* kept;       // [units][budget]
    int32_t* packed_lens;
    int* status;
    float* qnorm;        // [units][128], written by the select kernel
    float eps;
    int bf16;            // the window queries' type
    int scored;          // the kernel before the select is the second vote pass of this call
    int norm;            // the select kernel does the window norm too
};

template <typename E, int PASS>
__global__ void __launch_bounds__(kEvThreads) evict_scores_kernel(EvictArgs A)
{
    grid_wait();
    grid_release();
    extern __shared__ __align__(16) float ev_smem[];
    float* Ks = ev_smem;                                   // [128][129]
    float* Qs = Ks + kEvTile * kEvStride;                  // [64][129]
    float* colsum = Qs + kEvRows * kEvStride;              // [128]
    const int tile = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int S = min(A.seq_lens[b], A.S_max);
    if (S <= A.budget) return;                             // kept whole
    const int t0 = tile * kEvTile;
    if (t0 >= S) return;
    const int G = A.Hq / A.Hkv, R = G * A.W, P = S - A.W;
    const int unit = b * A.Hkv + h;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const float scale = rsqrtf(static_cast<float>(kHeadDim));

    for (int i = tid; i < kEvTile * kHeadDim; i += kEvThreads) {
        const int tt = i / kHeadDim, j = i - tt * kHeadDim;
        const int t = t0 + tt;
        Ks[tt * kEvStride + j] = (t < S)
            ? Elem<E>::load(A.k, static_cast<int64_t>(b) * A.sb + static_cast<int64_t>(h) * A.sh +
                                     static_cast<int64_t>(t) * A.st + j)
            : 0.f;
    }
    if (PASS == 2 && tid < kEvTile) colsum[tid] = 0.f;

    for (int r0 = 0; r0 < R; r0 += kEvRows) {
        __syncthreads();
        for (int i = tid; i < kEvRows * kHeadDim; i += kEvThreads) {
            const int rr = i / kHeadDim, j = i - rr * kHeadDim;
            const int row = r0 + rr;
            float v = 0.f;
            if (row < R) {
                const int g = row / A.W, w = row - g * A.W;
                v = Elem<E>::load(A.q_win, ((static_cast<int64_t>(b) * A.Hq + h * G + g) * A.W + w) * kHeadDim + j);
            }
            Qs[rr * kEvStride + j] = v;
        }
        __syncthreads();
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
        for (int kk = 0; kk < kHeadDim; ++kk) {
            float a[4], bb[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = Qs[(ty * 4 + i) * kEvStride + kk];
#pragma unroll
            for (int j = 0; j < 8; ++j) bb[j] = Ks[(tx + 16 * j) * kEvStride + kk];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
        }
        // thread (ty, tx): rows r0 + 4 ty + i, tokens t0 + tx + 16 j
        float cs[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) cs[j] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = r0 + ty * 4 + i;
            const bool row_ok = row < R;
            const int w = row_ok ? (row % A.W) : 0;
            const int last = P + w;                        // causal: this query sees tokens <= last
            if (PASS == 1) {
                float m = -INFINITY;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int t = t0 + tx + 16 * j;
                    acc[i][j] = (row_ok && t <= last && t < S) ? acc[i][j] * scale : -INFINITY;
                    m = fmaxf(m, acc[i][j]);
                }
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                float l = 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) l += (acc[i][j] == -INFINITY) ? 0.f : expf(acc[i][j] - m);
#pragma unroll
                for (int o = 1; o < 16; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
                if (row_ok && tx == 0) {
                    float* dst = A.partial + ((static_cast<int64_t>(unit) * R + row) * A.n_tiles + tile) * 2;
                    dst[0] = m;
                    dst[1] = l;
                }
            } else {
                float M = 0.f, invL = 0.f;
                if (row_ok) {
                    const float* rs = A.rowstat + (static_cast<int64_t>(unit) * R + row) * 2;
                    M = rs[0];
                    invL = 1.0f / rs[1];
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int t = t0 + tx + 16 * j;
                    if (row_ok && t < P) cs[j] += expf(acc[i][j] * scale - M) * invL;
                }
            }
        }
        if (PASS == 2) {
            // fixed-order accumulation of the column sums: row groups take turns
            for (int turn = 0; turn < 16; ++turn) {
                if (ty == turn)
#pragma unroll
                    for (int j = 0; j < 8; ++j) colsum[tx + 16 * j] += cs[j];
                __syncthreads();
            }
        }
    }
    if (PASS == 2) {
        __syncthreads();
        if (tid < kEvTile && t0 + tid < S)
            A.votes[static_cast<int64_t>(unit) * A.S_max + t0 + tid] = colsum[tid];
    }
}

__global__ void evict_rowstats_kernel(EvictArgs A)
{
    grid_wait();
    grid_release();
    const int h = blockIdx.x, b = blockIdx.y;
    const int S = min(A.seq_lens[b], A.S_max);
    if (S <= A.budget) return;
    const int G = A.Hq / A.Hkv, R = G * A.W;
    const int unit = b * A.Hkv + h;
    const int tiles = (S + kEvTile - 1) / kEvTile;
    for (int row = threadIdx.x; row < R; row += blockDim.x) {
        const float* src = A.partial + (static_cast<int64_t>(unit) * R + row) * A.n_tiles * 2;
        float M = -INFINITY, L = 0.f;
        for (int t = 0; t < tiles; ++t) {
            const float m = src[2 * t], l = src[2 * t + 1];
            if (m == -INFINITY) continue;
            const float Mn = fmaxf(M, m);
            L = L * expf(M - Mn) + l * expf(m - Mn);
            M = Mn;
        }
        A.rowstat[(static_cast<int64_t>(unit) * R + row) * 2] = M;
        A.rowstat[(static_cast<int64_t>(unit) * R + row) * 2 + 1] = L;
    }
}

// ------------------------------------------------------------------------------------------------
// Pooled votes, exact top-k and ordered compaction in ONE launch: a cluster of CTAs per (sequence, KV head), each with
// an equal share of the prefix.
//   pooled[t] = max of the votes within (pool-1)/2 positions of t (clamped to the prefix) as the float's bit pattern:
//   votes are >= 0, so unsigned comparison of the patterns is the order of the values.  The keys stay in the CTA's
//   shared memory (in the workspace where its share is larger than kKeyCap).
//   The k-th largest key is found by a radix select of 11 + 10 + 10 bits: every CTA histograms its keys in shared
//   memory, adds the non-empty bins to the first CTA's over distributed shared memory, and that CTA chooses.  (Every
//   CTA adding up all the histograms for itself was bound by those reads: 36 us with eight CTAs, 72 us with sixteen.)
//   Keys above the threshold, and the lowest positions among the equal ones, are written in order; a warp owns a
//   contiguous piece, and two counts per warp and CTA give it its place.
// What bounds it: dependent rounds over on-chip memory, a cluster barrier or two each.  As separate launches over all
// SMs (pool, four 8-bit histograms, count, compact) the 8 x 131072 keys of a prompt took 82 us under the profiler,
// this 22 us (four CTAs per unit: 30).  Keys in the workspace (1M tokens, two units) are asked for eight at a time: 393 us a
// prefill with one or four at a time, 336 so.
// ------------------------------------------------------------------------------------------------
constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelCluster = 8;             // CTAs per unit, at most (see select_cluster)
constexpr int kSelBatch = 8;               // keys a thread asks for at once where it has that many
constexpr int kVoteTile = 4 * kSelThreads; // raw votes staged at a time
constexpr int kVoteHalo = 256;             // widest pooling half that is staged
constexpr int kKeyCap = 36864;             // keys a CTA keeps in shared memory at most

// keys of one CTA for a prefix of P tokens (a multiple of the CTA's threads)
__host__ __device__ inline int select_share(int P, int ctas) { return (P + ctas * kSelThreads - 1) / (ctas * kSelThreads) * kSelThreads; }

// The bin (counted from the largest) that holds the need-th largest key, and the rank left inside it: v[] are the
// cluster's counts of this thread's kPer consecutive bins, largest bin first.
template <int kPer>
__device__ __forceinline__ void pick_bin(const int (&v)[kPer], int need, int tid, int* warp_sum, int* out)
{
    const int lane = tid & 31, warp = tid >> 5;
    int sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) sum += v[i];
    int inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int n = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += n; }
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    int before = __reduce_add_sync(0xffffffffu, lane < warp ? warp_sum[lane] : 0) + inc - sum;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        if (before < need && need <= before + v[i]) { out[0] = kPer * tid + i; out[1] = need - before; }
        before += v[i];
    }
}

__global__ void __launch_bounds__(kSelThreads) evict_select_kernel(EvictArgs A)
{
    extern __shared__ __align__(16) unsigned key_smem[];
    __shared__ int hist[2048 + 1024 + 1024], sums[2048 + 1024 + 1024];      // own counts; first CTA: the other CTAs'
    __shared__ int warp_sum[kSelWarps], warp_gt[kSelWarps], warp_eq[kSelWarps], total[2], pick[2];
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank()), ctas = gridDim.x, h = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* raw = reinterpret_cast<float*>(key_smem + A.key_cap);              // [kVoteTile + 2 * kVoteHalo]
    for (int i = tid; i < 4096; i += kSelThreads) hist[i] = sums[i] = 0;
    // The window norm of the unit, by the last CTA of its cluster (see norm_in_select): before the wait where the vote pass ran
    // (see grid_release).
    if (!A.scored) grid_wait();
    if (A.norm && rank == ctas - 1) {
        double (*part)[kHeadDim] = reinterpret_cast<double (*)[kHeadDim]>(key_smem);      // (at most 16 KB; the staging tile alone has 18)
        if (A.bf16) window_norm<__nv_bfloat16, 512>(A.q_win, A.Hq, A.Hkv, A.W, A.eps, A.qnorm, h, b, tid, part, [] {});
        else window_norm<float, 512>(A.q_win, A.Hq, A.Hkv, A.W, A.eps, A.qnorm, h, b, tid, part, [] {});
        __syncthreads();                                       // the keys go there next
    }
    if (A.scored) grid_wait();
    grid_release();
    int S = A.seq_lens[b];
    if (S < 0 || S > A.S_max) {
        if (rank == 0 && tid == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        S = S < 0 ? 0 : A.S_max;
    }
    const int unit = b * A.Hkv + h;
    int32_t* kept = A.kept + static_cast<int64_t>(unit) * A.budget;
    if (rank == 0 && h == 0 && tid == 0) A.packed_lens[b] = S < A.budget ? S : A.budget;
    if (S <= A.budget) {                                       // kept whole (the same in every CTA of the cluster)
        for (int t = rank * kSelThreads + tid; t < A.budget; t += ctas * kSelThreads) kept[t] = t < S ? t : -1;
        return;
    }
    const int P = S - A.W, k = A.budget - A.W, half = (A.pool - 1) / 2;
    if (rank == 0)
        for (int w = tid; w < A.W; w += kSelThreads) kept[k + w] = P + w;
    if (k == 0) return;                                        // the window alone
    const int share = select_share(P, ctas), c0 = rank * share;
    const int n = max(0, min(share, P - c0));                  // this CTA's keys: tokens c0 .. c0 + n - 1
    const int64_t base = static_cast<int64_t>(unit) * A.S_max;
    unsigned* keys = share <= A.key_cap ? key_smem : A.pooled + base + c0;
    const float* votes = A.votes + base;
    cluster.barrier_arrive();                                  // (waited for before the first CTA's sums, zeroed above, are added to)
    __syncthreads();
    // The raw votes come through a staging tile (with the pooling halo), the next tile's loads in flight while one is
    // pooled; very wide pools read the votes from memory.  A thread pools four neighbours; pooled neighbours are
    // mostly equal, so it counts runs of equal bins and most of the four cost no atomic of their own.
    const bool staged = half <= kVoteHalo;
    const int lead = staged ? half : 0;
    float next[kVoteTile / kSelThreads + 1];
    auto load_tile = [&](int i0) {
#pragma unroll
        for (int u = 0; u <= kVoteTile / kSelThreads; ++u) {
            const int x = u * kSelThreads + tid, t = c0 + i0 - lead + x;
            next[u] = (x < kVoteTile + 2 * lead && t >= 0 && t < P) ? votes[t] : 0.f;      // votes are >= 0
        }
    };
    load_tile(0);
    for (int i0 = 0; i0 < share; i0 += kVoteTile) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u <= kVoteTile / kSelThreads; ++u) {
            const int x = u * kSelThreads + tid;
            if (x < kVoteTile + 2 * lead) raw[x] = next[u];
        }
        __syncthreads();
        if (i0 + kVoteTile < share) load_tile(i0 + kVoteTile);
        const int x = 4 * tid, i = i0 + x;
        if (i < n) {
            float m[4];
            if (half == 3) {
                const float4 r0 = *reinterpret_cast<const float4*>(raw + x), r1 = *reinterpret_cast<const float4*>(raw + x + 4);
                const float2 r2 = *reinterpret_cast<const float2*>(raw + x + 8);
                const float mid = fmaxf(fmaxf(r0.w, r1.x), fmaxf(r1.y, r1.z));           // in all four windows
                const float yz = fmaxf(r0.y, r0.z), ab = fmaxf(r1.w, r2.x);
                m[0] = fmaxf(mid, fmaxf(r0.x, yz));
                m[1] = fmaxf(mid, fmaxf(yz, r1.w));
                m[2] = fmaxf(mid, fmaxf(r0.z, ab));
                m[3] = fmaxf(mid, fmaxf(ab, r2.y));
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    m[e] = raw[x + e + lead];
                    if (staged) {
                        for (int u = 0; u <= 2 * half; ++u) m[e] = fmaxf(m[e], raw[x + e + u]);
                    } else {
                        for (int u = max(0, c0 + i + e - half); u <= min(P - 1, c0 + i + e + half); ++u) m[e] = fmaxf(m[e], votes[u]);
                    }
                }
            }
            int run = 0, bin = 0;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (i + e < n) {
                    const unsigned key = __float_as_uint(m[e]);
                    keys[i + e] = key;
                    const int bn = (key >> 20) & 2047u;
                    if (run && bn != bin) { atomicAdd(&hist[bin], run); run = 0; }
                    bin = bn;
                    ++run;
                }
            }
            atomicAdd(&hist[bin], run);
        }
    }
    // One pass of the radix select over the bins hp (this CTA) and sum (first CTA): x the chosen bin, y the rank inside it
    auto choose = [&](int* hp, int* sum, auto per, int want, bool first) {
        constexpr int kPer = decltype(per)::value, kBins = kPer * kSelThreads;
        __syncthreads();
        if (first) cluster.barrier_wait();
        if (rank > 0) {
            int* to = cluster.map_shared_rank(sum, 0);
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int c = hp[u * kSelThreads + tid];
                if (c) atomicAdd(to + u * kSelThreads + tid, c);
            }
        }
        cluster.sync();
        if (rank == 0) {
            int v[kPer];
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int bin = kBins - 1 - (kPer * tid + u);
                v[u] = hp[bin] + sum[bin];
            }
            pick_bin<kPer>(v, want, tid, warp_sum, pick);
        }
        cluster.sync();
        const int* choice = cluster.map_shared_rank(pick, 0);
        return make_int2(kBins - 1 - choice[0], choice[1]);
    };
    int2 c = choose(hist, sums, std::integral_constant<int, 2>(), k, true);
    unsigned thr = static_cast<unsigned>(c.x) << 20;
    int need = c.y;
#pragma unroll 1
    for (int pass = 1; pass < 3; ++pass) {
        const int shift = pass == 1 ? 10 : 0;
        int* hp = hist + 1024 + 1024 * pass;
        const unsigned top = thr >> (shift + 10);
        auto count = [&](unsigned key) { if ((key >> (shift + 10)) == top) atomicAdd(&hp[(key >> shift) & 1023u], 1); };
        int i = tid;
        for (; i + (kSelBatch - 1) * kSelThreads < n; i += kSelBatch * kSelThreads) {
            unsigned key[kSelBatch];
#pragma unroll
            for (int u = 0; u < kSelBatch; ++u) key[u] = keys[i + u * kSelThreads];
#pragma unroll
            for (int u = 0; u < kSelBatch; ++u) count(key[u]);
        }
        for (; i < n; i += kSelThreads) count(keys[i]);
        c = choose(hp, sums + 1024 + 1024 * pass, std::integral_constant<int, 1>(), need, false);
        thr |= static_cast<unsigned>(c.x) << shift;
        need = c.y;
    }
    // keys above / equal to the threshold, per warp (a contiguous piece each) and per CTA
    const int seg = share / kSelWarps, s0 = warp * seg;
    int gt = 0, eq = 0;
    const int s1 = min(n, s0 + seg);                           // (the same in every lane)
    auto above = [&](unsigned key) { gt += key > thr; eq += key == thr; };
    {
        int i = s0 + lane;
        for (; i - lane + 32 * kSelBatch <= s1; i += 32 * kSelBatch) {
            unsigned key[kSelBatch];
#pragma unroll
            for (int u = 0; u < kSelBatch; ++u) key[u] = keys[i + 32 * u];
#pragma unroll
            for (int u = 0; u < kSelBatch; ++u) above(key[u]);
        }
        for (; i < s1; i += 32) above(keys[i]);
    }
    gt = __reduce_add_sync(0xffffffffu, gt);
    eq = __reduce_add_sync(0xffffffffu, eq);
    if (lane == 0) { warp_gt[warp] = gt; warp_eq[warp] = eq; }
    __syncthreads();
    int b_gt = __reduce_add_sync(0xffffffffu, lane < warp ? warp_gt[lane] : 0);        // before this warp's piece
    int b_eq = __reduce_add_sync(0xffffffffu, lane < warp ? warp_eq[lane] : 0);
    if (tid == kSelThreads - 1) { total[0] = b_gt + gt; total[1] = b_eq + eq; }
    cluster.sync();
    int own_gt = 0;
    for (int r = 0; r < rank; ++r) {
        const int* t = cluster.map_shared_rank(total, r);
        own_gt += t[0]; b_eq += t[1];
    }
    if (rank == ctas - 1 && tid == 0 && own_gt + total[0] + need != k) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
    b_gt += own_gt;
    const unsigned lt = (1u << lane) - 1u;
    auto place = [&](int i, bool on, unsigned key) {           // the warp's keys at i - lane .. i - lane + 31
        const unsigned mg = __ballot_sync(0xffffffffu, on && key > thr), me = __ballot_sync(0xffffffffu, on && key == thr);
        const int eq_rank = b_eq + __popc(me & lt);            // equal keys on lower positions
        const int pos = b_gt + __popc(mg & lt) + min(eq_rank, need);
        if (((mg >> lane) & 1u) || (((me >> lane) & 1u) && eq_rank < need)) {
            if (pos < k) kept[pos] = c0 + i;
        }
        b_gt += __popc(mg);
        b_eq += __popc(me);
    };
    int i0 = s0;
    for (; i0 + 32 * kSelBatch <= s1; i0 += 32 * kSelBatch) {
        unsigned key[kSelBatch];
#pragma unroll
        for (int u = 0; u < kSelBatch; ++u) key[u] = keys[i0 + 32 * u + lane];
#pragma unroll
        for (int u = 0; u < kSelBatch; ++u) place(i0 + 32 * u + lane, true, key[u]);
    }
    for (; i0 < s1; i0 += 32) place(i0 + lane, i0 + lane < s1, i0 + lane < s1 ? keys[i0 + lane] : 0u);
    cluster.sync();                                            // the others may still be reading this CTA's totals
}

// CTAs per unit (a power of two).  A barrier of the cluster costs more than the keys it spares a CTA below some 8000, and a
// cluster of 1024-thread CTAs that does not fit beside the others waits for a whole second round: 64 x 1500 tokens with 8 KV
// heads (512 units) took 559 us an evicting prefill with eight CTAs per unit and takes 268 with one, 4 x 8000 85.5 and 66;
// with 16 units of 60000 four are better than eight (156 against 164), with four units of 32768 or 131072 eight (67.5, 188)
// than four (69.5, 199).  Very wide pools are bound by their pooling, which wants every SM.
inline int select_cluster(int64_t units, int prefix, int pool)
{
    if (pool > 64) return kSelCluster;
    int c = prefix <= 8192 ? 1 : (units <= 12 ? 8 : (units <= 32 ? 4 : (units <= 64 ? 2 : 1)));
    while (c < kSelCluster && select_share(prefix, c) > kKeyCap) c *= 2;  // the keys stay on chip if they can
    return c;
}

bool evict_tc_supported(const spark_params& p);
spark_status launch_evict_votes_tc(const spark_params& p, const void* q_win, const void* k, int64_t sb, int64_t sh,
                                   int64_t st, const int32_t* seq_lens, int32_t max_seq_tokens, float* partial,
                                   float* votes, int* status, cudaStream_t stream, int* launches, bool* done);

size_t evict_workspace_bytes(const spark_params& p, int64_t max_seq_tokens)
{
    if (p.token_budget <= 0) return 0;
    const size_t units = static_cast<size_t>(p.batch) * p.n_kv_heads;
    const size_t R = static_cast<size_t>(p.n_q_heads / p.n_kv_heads) * p.window;
    const size_t tiles = (max_seq_tokens + kEvTile - 1) / kEvTile;
    size_t bytes = units * R * tiles * 2 * sizeof(float);
    bytes += units * R * 2 * sizeof(float);
    bytes += 2 * units * static_cast<size_t>(max_seq_tokens) * sizeof(float);      // votes, pooled keys
    return (bytes + 255) / 256 * 256;
}

spark_status launch_evict(const spark_params& p, const void* q_win, const void* k, int64_t sb, int64_t sh,
                          int64_t st, const int32_t* seq_lens, int32_t max_seq_tokens, float* qnorm, int32_t* packed_lens,
                          int32_t* kept_tokens, void* workspace, cudaStream_t stream, int* launches)
{
    const size_t units = static_cast<size_t>(p.batch) * p.n_kv_heads;
    const size_t R = static_cast<size_t>(p.n_q_heads / p.n_kv_heads) * p.window;
    EvictArgs A;
    A.q_win = q_win; A.k = k; A.sb = sb; A.sh = sh; A.st = st; A.seq_lens = seq_lens;
    A.Hq = p.n_q_heads; A.Hkv = p.n_kv_heads; A.W = p.window; A.budget = p.token_budget; A.pool = p.pool_kernel;
    A.S_max = max_seq_tokens; A.n_tiles = (max_seq_tokens + kEvTile - 1) / kEvTile;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    A.status = reinterpret_cast<int*>(ws);
    A.partial = reinterpret_cast<float*>(ws + kWorkspaceHeader);
    A.rowstat = A.partial + units * R * A.n_tiles * 2;
    A.votes = A.rowstat + units * R * 2;
    A.pooled = reinterpret_cast<unsigned*>(A.votes + units * static_cast<size_t>(max_seq_tokens));
    A.kept = kept_tokens; A.packed_lens = packed_lens;
    const size_t smem = (static_cast<size_t>(kEvTile + kEvRows) * kEvStride + kEvTile) * sizeof(float);
    const dim3 grid(A.n_tiles, p.n_kv_heads, p.batch), ugrid(p.n_kv_heads, p.batch);
    const bool bf16 = p.dtype == SPARK_BF16;
    A.qnorm = qnorm; A.eps = norm_floor(p); A.bf16 = bf16; A.norm = norm_in_select(static_cast<int64_t>(units));
    A.scored = A.n_tiles > 0 && max_seq_tokens > p.token_budget;
    // (the tensor-core kernels read the window queries 16 bytes at a time; the call does not ask for that alignment)
    const bool q_aligned = (reinterpret_cast<uintptr_t>(q_win) & 15) == 0;
    bool voted = !A.scored;
    if (A.scored && q_aligned && evict_tc_supported(p)) {
        const spark_status st_tc = launch_evict_votes_tc(p, q_win, k, sb, sh, st, seq_lens, max_seq_tokens, A.partial,
                                                         A.votes, A.status, stream, launches, &voted);
        if (st_tc != SPARK_OK) return st_tc;
    }
    if (!voted) {
        static unsigned char smem_raised[4][kMaxDevices] = {};
        if (!(bf16 ? allow_max_smem(evict_scores_kernel<__nv_bfloat16, 1>, smem_raised[0]) && allow_max_smem(evict_scores_kernel<__nv_bfloat16, 2>, smem_raised[1])
                   : allow_max_smem(evict_scores_kernel<float, 1>, smem_raised[2]) && allow_max_smem(evict_scores_kernel<float, 2>, smem_raised[3])))
            return SPARK_ERR_CUDA;
        if (bf16) launch_kernel(evict_scores_kernel<__nv_bfloat16, 1>, grid, dim3(kEvThreads), smem, stream, A);
        else launch_kernel(evict_scores_kernel<float, 1>, grid, dim3(kEvThreads), smem, stream, A);
        launch_kernel(evict_rowstats_kernel, ugrid, dim3(256), 0, stream, A);
        if (bf16) launch_kernel(evict_scores_kernel<__nv_bfloat16, 2>, grid, dim3(kEvThreads), smem, stream, A);
        else launch_kernel(evict_scores_kernel<float, 2>, grid, dim3(kEvThreads), smem, stream, A);
        *launches += 3;
    }
    DeviceInfo info;
    int dev = 0;
    if (!device_info(&dev, &info)) return SPARK_ERR_CUDA;
    const int prefix = max_seq_tokens > p.window ? max_seq_tokens - p.window : 1;
    const int ctas = select_cluster(static_cast<int64_t>(units), prefix, p.pool_kernel);
    const int most = select_share(prefix, ctas);
    A.key_cap = most < kKeyCap ? most : kKeyCap;
    const size_t key_bytes = (static_cast<size_t>(A.key_cap) + kVoteTile + 2 * kVoteHalo) * sizeof(unsigned);
    static unsigned char select_raised[kMaxDevices] = {};
    if (!allow_max_smem(evict_select_kernel, dev, info.smem_optin, select_raised)) return SPARK_ERR_CUDA;
    launch_cluster(evict_select_kernel, ctas, dim3(ctas, p.n_kv_heads, p.batch), dim3(kSelThreads), key_bytes, stream, A);
    ++*launches;
    return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace spark
