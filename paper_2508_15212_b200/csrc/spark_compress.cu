// Prefill-side kernels: window-mean query norm, per-token top-T channel selection + page packing,
// and the inverse (pages -> logical arrays).
//
// Method (paper sections): the mean window query replaces per-token queries (Sec. "SparK"); the
// saliency of channel j of token t is w = |q-bar_j| * |K[t][j]| (Sec. "Problem Formulation"); the T
// channels of largest w are kept (Eq. (cal)); the mean saliency of the pruned channels is cached per
// token (App. "Caching Pruned Channel Statistics").  With value-channel pruning (App. "Pruning Value
// Cache Channels") the same per-token selection runs on |V[t][j]| and the page stores the kept values and a
// second mask instead of the dense value row.
#include <type_traits>

#include "spark_common.cuh"

namespace spark {

constexpr unsigned kFullMask = 0xffffffffu;

// ------------------------------------------------------------------------------------------------
// The window norm (window_norm) as a launch of its own; with eviction and few units the select kernel does it (norm_in_select).  128 to 512 threads
// (qnorm_threads).  The chain that bounds it is a load and a few adds: one thread per channel walking all rows took 8.3 us for
// 128 rows, this 7.1 (both cold), and the page kernel's first loads run under it.
// Thread 0 of the first head also publishes packed_lens (where there is no eviction).
// ------------------------------------------------------------------------------------------------
template <typename E, int kThreads, bool kReleaseEarly>
__global__ void __launch_bounds__(kThreads)
window_qnorm_kernel(const void* __restrict__ q_win, int Hq, int Hkv, int W, float eps,
                    float* __restrict__ qnorm, const int32_t* __restrict__ seq_lens,
                    int32_t* __restrict__ packed_lens, int max_seq_tokens, int* status)
{
    constexpr int kGroups = kThreads / (kHeadDim / (16 / static_cast<int>(sizeof(E))));
    __shared__ double part[kGroups / 2][kHeadDim];
    grid_wait();
    if (kReleaseEarly) grid_release();
    const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
    window_norm<E, kThreads>(q_win, Hq, Hkv, W, eps, qnorm, h, b, tid, part, [] { if (!kReleaseEarly) grid_release(); });
    if (packed_lens && h == 0 && tid == 0) {
        int len = seq_lens[b];
        if (len < 0 || len > max_seq_tokens) {
            record_error(status, SPARK_ERR_DEVICE_BOUNDS);
            len = len < 0 ? 0 : max_seq_tokens;
        }
        packed_lens[b] = len;
    }
}

// ------------------------------------------------------------------------------------------------
// One token of one KV head, one warp: saliency, exact top-T selection, and the token's entries of a
// page image at `image` (kept values in slot order, mask words, mu).  A lane owns channels
// 4*lane .. 4*lane+3: `kf` are its key values, `raw` their stored bit patterns, `a` its qnorm entries.
//
// Selection is exact: the saliency is one __fmul_rn, its bit pattern (non-negative float) is an
// order-preserving 31-bit key, the T-th largest key is found by a bitwise radix descent with warp
// reductions, and keys equal to it are admitted in ascending channel order until T channels are kept.
//
// The same routine prunes a value row (a = 1, so the key is |V[t][j]| itself): `vals_off` / `mask_off`
// select the section that receives the kept entries and the mask, and mu is written only when
// `mu_off` >= 0 (`inv_pruned` = 1 / (D - T), or 0 when nothing is pruned: the mean is taken as a product
// in double, which rounds to the same float as the quotient except on a rounding boundary of the double).
// ------------------------------------------------------------------------------------------------
// How the kept key channels of a token are chosen, and which statistics the page stores.
struct SelectArgs {
    int select;                   // spark_select
    float top_p;                  // SPARK_SELECT_TOP_P
    unsigned rank_keep[4];        // SPARK_SELECT_GROUPS: bit r set <=> the channel of saliency rank r is kept
    int recovery;                 // spark_recovery: a sampled distribution needs the all-channel statistics
};

// Exact top-T of the warp's 128 keys: kept[i] for the lane's four channels (see pack_token).
__device__ __forceinline__ void select_top_t(const unsigned (&key)[4], int T, int lane, bool (&kept)[4])
{
    const unsigned lt = (1u << lane) - 1u;
    // T-th largest key by radix descent over the bits in which the 128 keys differ.  The descent
    // stops as soon as a candidate threshold has exactly T keys at or above it (then those are the
    // kept set and no tie can straddle the boundary); otherwise it ends with the exact T-th largest
    // key and equal keys are admitted in ascending channel order.
    const unsigned k_or = __reduce_or_sync(kFullMask, key[0] | key[1] | key[2] | key[3]);
    const unsigned k_and = __reduce_and_sync(kFullMask, key[0] & key[1] & key[2] & key[3]);
    const unsigned diff = k_or ^ k_and;
    const int top = diff ? (31 - __clz(diff)) : -1;              // highest bit in which keys differ
    unsigned thr = (top >= 0) ? (k_and & ~((2u << top) - 1u)) : k_and;   // common leading bits
    bool exact = false;
    for (int bit = top; bit >= 0; --bit) {
        const unsigned cand = thr | (1u << bit);
        const int mine = (key[0] >= cand) + (key[1] >= cand) + (key[2] >= cand) + (key[3] >= cand);
        const int cnt = __reduce_add_sync(kFullMask, mine);
        if (cnt >= T) thr = cand;
        if (cnt == T) { exact = true; break; }
    }
    if (exact) {
#pragma unroll
        for (int i = 0; i < 4; ++i) kept[i] = key[i] >= thr;
    } else {
        unsigned eqb[4];
        int c_gt = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            c_gt += __popc(__ballot_sync(kFullMask, key[i] > thr));
            eqb[i] = __ballot_sync(kFullMask, key[i] == thr);
        }
        const int need_eq = T - c_gt;
        int rank = 0;                                        // equal keys on lower channels
#pragma unroll
        for (int i = 0; i < 4; ++i) rank += __popc(eqb[i] & lt);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool eq = key[i] == thr;
            kept[i] = key[i] > thr || (eq && rank < need_eq);
            rank += eq ? 1 : 0;
        }
    }
}

// The ratio-free selection rules (Sec. "Ablation Studies", adaptive variants) need every channel's saliency
// RANK, so the warp sorts its 128 keys: a bitonic network over (saliency bits, 127 - channel), descending,
// four consecutive ranks per lane.  SparK-p then keeps the shortest rank prefix whose saliencies (summed in
// double, most salient first) reach top_p of the token's total, at least one and at most `cap` channels;
// SparK-g keeps the ranks listed in rank_keep.  Returns kept[i] for the lane's four CHANNELS and the count.
__device__ __forceinline__ int select_by_rank(const unsigned (&key)[4], int lane, const SelectArgs& sel, int cap,
                                              bool (&kept)[4])
{
    unsigned long long K[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        K[e] = (static_cast<unsigned long long>(key[e]) << 7) | static_cast<unsigned>(127 - (4 * lane + e));
#pragma unroll
    for (int size = 2; size <= 128; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 4) {
                const bool lower = ((4 * lane) & stride) == 0;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const unsigned long long other = __shfl_xor_sync(kFullMask, K[e], stride >> 2);
                    const bool down = ((4 * lane + e) & size) == 0;     // this block ends up descending
                    const bool take_max = (lower == down);
                    K[e] = take_max ? (K[e] > other ? K[e] : other) : (K[e] < other ? K[e] : other);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if ((e & stride) == 0) {
                        const bool down = ((4 * lane + e) & size) == 0;
                        const unsigned long long x = K[e], y = K[e ^ stride];
                        const unsigned long long hi = x > y ? x : y, lo = x > y ? y : x;
                        K[e] = down ? hi : lo;
                        K[e ^ stride] = down ? lo : hi;
                    }
            }
        }
    }
    unsigned rk[4] = {sel.rank_keep[0], sel.rank_keep[1], sel.rank_keep[2], sel.rank_keep[3]};
    if (sel.select == SPARK_SELECT_TOP_P) {
        double c[4];
        double run = 0.0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            run += static_cast<double>(__uint_as_float(static_cast<unsigned>(K[e] >> 7)));
            c[e] = run;
        }
        double incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double up = __shfl_up_sync(kFullMask, incl, o);
            if (lane >= o) incl += up;
        }
        const double total = __shfl_sync(kFullMask, incl, 31);
        const double need = static_cast<double>(sel.top_p) * total;
        const double before = incl - run;
        int below = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) below += (before + c[e] < need) ? 1 : 0;
        int n = __reduce_add_sync(kFullMask, below) + 1;       // first rank whose running sum reaches `need`
        n = n > kHeadDim ? kHeadDim : n;
        n = n > cap ? cap : n;
#pragma unroll
        for (int wi = 0; wi < 4; ++wi)
            rk[wi] = n >= 32 * (wi + 1) ? 0xffffffffu : (n > 32 * wi ? ((1u << (n - 32 * wi)) - 1u) : 0u);
    }
    unsigned m[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int r = 4 * lane + e;
        if ((rk[r >> 5] >> (r & 31)) & 1u) {
            const int j = 127 - static_cast<int>(K[e] & 127u);
#pragma unroll
            for (int wi = 0; wi < 4; ++wi)
                if ((j >> 5) == wi) m[wi] |= 1u << (j & 31);
        }
    }
    int n_kept = 0;
#pragma unroll
    for (int wi = 0; wi < 4; ++wi) {
        m[wi] = __reduce_or_sync(kFullMask, m[wi]);
        n_kept += __popc(m[wi]);
    }
    unsigned mine = m[0];
#pragma unroll
    for (int wi = 1; wi < 4; ++wi)
        if ((lane >> 3) == wi) mine = m[wi];
#pragma unroll
    for (int i = 0; i < 4; ++i) kept[i] = (mine >> (4 * (lane & 7) + i)) & 1u;
    return n_kept;
}

template <bool kBf16, bool kRank>
__device__ __forceinline__ int pack_token(unsigned char* image, int vals_off, int mask_off, int mu_off,
                                           int p, int T, int lane,
                                           const float (&a)[4], const float (&kf)[4], const unsigned (&raw)[4],
                                           double inv_pruned = 0.0, const SelectArgs* sel = nullptr, int stats_off = -1)
{
    const unsigned lt = (1u << lane) - 1u;
    float w[4];
    unsigned key[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        w[i] = __fmul_rn(a[i], fabsf(kf[i]));                 // the one rounding that decides selection
        key[i] = __float_as_uint(w[i]);
    }
    bool kept[4];
    int n_kept = T;
    if (kRank) n_kept = select_by_rank(key, lane, *sel, T, kept);     // a ratio-free rule (keys only)
    else select_top_t(key, T, lane, kept);
    // slot of each kept channel = kept channels below it
    int slot = 0;
    unsigned nib = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        slot += __popc(__ballot_sync(kFullMask, kept[i]) & lt);
        nib |= kept[i] ? (1u << i) : 0u;
    }
    double pruned = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (kept[i]) {
            unsigned char* dst = image + vals_off + val_offset(kBf16 ? 2 : 4, p, slot);
            if (kBf16) *reinterpret_cast<unsigned short*>(dst) = static_cast<unsigned short>(raw[i]);
            else *reinterpret_cast<unsigned*>(dst) = raw[i];
            ++slot;
        } else {
            pruned += static_cast<double>(w[i]);
        }
    }
    unsigned word = nib << (4 * (lane & 7));
    word |= __shfl_xor_sync(kFullMask, word, 1);
    word |= __shfl_xor_sync(kFullMask, word, 2);
    word |= __shfl_xor_sync(kFullMask, word, 4);
    if ((lane & 7) == 0)
        reinterpret_cast<unsigned*>(image + mask_off)[p * kMaskWords + (lane >> 3)] = word;
    if (mu_off < 0) return n_kept;                            // warp-uniform
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pruned += __shfl_xor_sync(kFullMask, pruned, o);
    if (lane == 0) {
        float mu;
        if (kRank)
            mu = n_kept < kHeadDim ? static_cast<float>(pruned / static_cast<double>(kHeadDim - n_kept)) : 0.f;
        else
            mu = static_cast<float>(pruned * inv_pruned);
        reinterpret_cast<float*>(image + mu_off)[p] = mu;
    }
    if (stats_off < 0) return n_kept;                         // warp-uniform
    // all-channel mean and population deviation of the token's saliencies (sampled recovery)
    double s1 = (static_cast<double>(w[0]) + static_cast<double>(w[1])) + (static_cast<double>(w[2]) + static_cast<double>(w[3]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s1 += __shfl_xor_sync(kFullMask, s1, o);
    const double mean = s1 / static_cast<double>(kHeadDim);
    double s2 = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) { const double d = static_cast<double>(w[i]) - mean; s2 += d * d; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(kFullMask, s2, o);
    if (lane == 0) {
        reinterpret_cast<float*>(image + stats_off)[p] = static_cast<float>(mean);
        reinterpret_cast<float*>(image + stats_off)[kPageTokens + p] = static_cast<float>(sqrt(s2 / static_cast<double>(kHeadDim)));
    }
    return n_kept;
}

// Key entries and value entries of one token row into the page image.  A lane owns channels 4*lane ..
// 4*lane+3; `row` is the element offset of its first channel in k and v.  `inv_pruned` = 1 / (D - T)
// (0 when T = D), computed once on the host.
template <bool kBf16, bool kRank>
__device__ __forceinline__ int pack_token_kv(unsigned char* image, const PageLayout& L, int p, int lane,
                                              const float (&a)[4], const void* k, const void* v, int64_t row,
                                              double inv_pruned, const SelectArgs& sel)
{
    unsigned kraw[4], vraw[4];
    float kf[4];
    if (kBf16) {
        const uint2 kk = *reinterpret_cast<const uint2*>(static_cast<const unsigned short*>(k) + row);
        const uint2 vv = *reinterpret_cast<const uint2*>(static_cast<const unsigned short*>(v) + row);
        kraw[0] = kk.x & 0xffffu; kraw[1] = kk.x >> 16; kraw[2] = kk.y & 0xffffu; kraw[3] = kk.y >> 16;
#pragma unroll
        for (int i = 0; i < 4; ++i) kf[i] = __uint_as_float(kraw[i] << 16);
        if (L.keep_v < kHeadDim) {
            vraw[0] = vv.x & 0xffffu; vraw[1] = vv.x >> 16; vraw[2] = vv.y & 0xffffu; vraw[3] = vv.y >> 16;
        } else {
            *reinterpret_cast<uint2*>(image + L.v_off + v_chunk_offset(2, p, lane >> 1) + (lane & 1) * 8) = vv;
        }
    } else {
        const uint4 kk = *reinterpret_cast<const uint4*>(static_cast<const float*>(k) + row);
        const uint4 vv = *reinterpret_cast<const uint4*>(static_cast<const float*>(v) + row);
        kraw[0] = kk.x; kraw[1] = kk.y; kraw[2] = kk.z; kraw[3] = kk.w;
#pragma unroll
        for (int i = 0; i < 4; ++i) kf[i] = __uint_as_float(kraw[i]);
        if (L.keep_v < kHeadDim) { vraw[0] = vv.x; vraw[1] = vv.y; vraw[2] = vv.z; vraw[3] = vv.w; }
        else *reinterpret_cast<uint4*>(image + L.v_off + v_chunk_offset(4, p, lane)) = vv;
    }
    if (L.keep_v < kHeadDim) {                             // value-channel pruning: same selection on |V|
        float vf[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) vf[i] = __uint_as_float(kBf16 ? vraw[i] << 16 : vraw[i]);
        const float one[4] = {1.f, 1.f, 1.f, 1.f};
        pack_token<kBf16, false>(image, L.v_off, L.vmask_off, -1, p, L.keep_v, lane, one, vf, vraw);
    }
    return pack_token<kBf16, kRank>(image, L.vals_off, L.mask_off, L.mu_off, p, L.keep, lane, a, kf, kraw, inv_pruned, &sel,
                             L.recovery != SPARK_RECOVER_DEGENERATE ? L.stats_off : -1);
}

// ------------------------------------------------------------------------------------------------
// The ratio-free rules that sort (SparK-g; SparK-p on fp32 storage, with pruned values or sampled recovery): one CTA builds
// one page (16 tokens of one KV head) in shared memory and writes it out with coalesced 16-byte stores.  One warp per token,
// two rounds; a lane owns channels 4*lane .. 4*lane+3; keys are chosen by select_by_rank, pruned values by select_top_t.
// ------------------------------------------------------------------------------------------------
struct CompressArgs {
    const void* k;
    const void* v;
    int64_t sb, sh, st;
    const int32_t* lens;          // tokens per sequence AFTER eviction (packed lens)
    int max_len;                  // upper bound of lens (compress_pages_warp_kernel reads the caller's lengths, unchecked)
    const int32_t* gather;        // optional [B][Hkv][gather_stride] source token positions
    int gather_stride;
    const float* qnorm;
    unsigned char* pages;
    const int32_t* block_table;
    int max_blocks;
    int Hkv;
    int keep;
    int64_t n_pool_pages;
    PageLayout L;
    double inv_pruned;            // 1 / (D - T), 0 when T = D
    SelectArgs sel;
    int* status;
};

template <typename E>
__global__ void __launch_bounds__(256) compress_pages_kernel(CompressArgs A)
{
    grid_wait();
    grid_release();
    extern __shared__ __align__(16) unsigned char image[];
    const int blk = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int len = A.lens[b];
    if (blk * kPageTokens >= len) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const PageLayout L = A.L;
    constexpr bool kBf16 = (sizeof(E) == 2);

    __shared__ int rows_used;
    if (threadIdx.x == 0) rows_used = 0;
    for (int i = threadIdx.x; i < L.page_bytes / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(image)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    const float4 a4 = reinterpret_cast<const float4*>(
        A.qnorm + (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim)[lane];
    const float a[4] = {a4.x, a4.y, a4.z, a4.w};
    for (int p = warp; p < kPageTokens; p += 8) {
        const int t = blk * kPageTokens + p;
        if (t >= len) continue;                                   // warp-uniform
        const int src_t = A.gather
            ? A.gather[(static_cast<int64_t>(b) * A.Hkv + h) * A.gather_stride + t] : t;
        const int64_t row = static_cast<int64_t>(b) * A.sb + static_cast<int64_t>(h) * A.sh +
                            static_cast<int64_t>(src_t) * A.st + lane * 4;
        const int n_kept = pack_token_kv<kBf16, true>(image, L, p, lane, a, A.k, A.v, row, A.inv_pruned, A.sel);
        if (L.ragged && lane == 0) atomicMax(&rows_used, n_kept);
    }
    __syncthreads();

    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    const int64_t page_id = A.block_table ? A.block_table[entry] : entry;     // no table: contiguous cache
    if (page_id < 0 || page_id >= A.n_pool_pages) {
        if (threadIdx.x == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    uint4* dst = reinterpret_cast<uint4*>(A.pages + page_id * L.page_bytes);
    for (int i = threadIdx.x; i < L.page_bytes / 16; i += blockDim.x)
        dst[i] = reinterpret_cast<const uint4*>(image)[i];
    if (L.ragged && threadIdx.x == 0)
        reinterpret_cast<int*>(A.pages + rows_offset(A.n_pool_pages, L.page_bytes))[page_id] = rows_used;
}

// ------------------------------------------------------------------------------------------------
// Fixed-T pages of fp32 storage and of sampled recovery, four tokens per warp.  Most of what the selection costs per token is warp-wide
// bookkeeping (reductions, votes, loop control) that serves one token when a warp owns one token.  Here a
// token belongs to EIGHT lanes (16 channels per lane), a warp carries four tokens through the same
// instructions, and the radix descent compares two keys per instruction while it works on the keys' upper
// 16 bits (the bf16 image of a non-negative float orders like the float): a compare yields 1.0 or
// 0 per key, and the ones are added in half precision (at most 8 a half: exact).  Below bit 16 the descent continues on the
// full keys.  The result is the same exact top-T set, with ties to the lower channel, as select_top_t.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int group8_sum(int v)              // (a masked hardware reduction measured slower)
{
    v += __shfl_xor_sync(kFullMask, v, 1);
    v += __shfl_xor_sync(kFullMask, v, 2);
    v += __shfl_xor_sync(kFullMask, v, 4);
    return v;
}
__device__ __forceinline__ double group8_sum(double v)
{
    v += __shfl_xor_sync(kFullMask, v, 1);
    v += __shfl_xor_sync(kFullMask, v, 2);
    v += __shfl_xor_sync(kFullMask, v, 4);
    return v;
}
__device__ __forceinline__ int group8_exclusive(int v, int l8)      // sum over the lower lanes of the group
{
    int x = v;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const int y = __shfl_up_sync(kFullMask, x, o, 8);
        if (l8 >= o) x += y;
    }
    return x - v;
}
// per half: 1.0 (bf16) where a >= b, else 0 -- on the half-precision pipe, so that counting the keys at or
// above a candidate costs the integer pipe nothing
__device__ __forceinline__ __nv_bfloat162 ge_one_bf16x2(unsigned a, unsigned b)
{
    return __hge2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
}

// kept bits (bit i <=> the lane's channel i) of the exact top-T among the 128 keys of the lane's group
__device__ __forceinline__ unsigned select_top_t16(const unsigned (&key)[16], int T, int l8)
{
    unsigned hk[8];                                              // upper halves of the keys, two per word
#pragma unroll
    for (int i = 0; i < 8; ++i) hk[i] = (key[2 * i] >> 16) | (key[2 * i + 1] & 0xffff0000u);
    // bits in which the group's keys differ: from the upper halves, and from the full keys only when the
    // upper halves all agree
    unsigned o = hk[0], n = hk[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) { o |= hk[i]; n &= hk[i]; }
    o |= o << 16; n &= n << 16;                                  // fold the two keys of a word into the upper half
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) {
        o |= __shfl_xor_sync(kFullMask, o, d);
        n &= __shfl_xor_sync(kFullMask, n, d);
    }
    o &= 0xffff0000u; n &= 0xffff0000u;
    if (__any_sync(kFullMask, o == n)) {                         // rare: some group's keys share their upper halves
        unsigned o2 = key[0], n2 = key[0];
#pragma unroll
        for (int i = 1; i < 16; ++i) { o2 |= key[i]; n2 &= key[i]; }
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) {
            o2 |= __shfl_xor_sync(kFullMask, o2, d);
            n2 &= __shfl_xor_sync(kFullMask, n2, d);
        }
        o = o2; n = n2;
    } else {
        o |= 0xffffu;                                            // lower halves: treated as differing everywhere
    }
    const unsigned diff = o ^ n;
    const int top = diff ? (31 - __clz(diff)) : -1;              // highest bit in which the group's keys differ
    unsigned thr = (top >= 0) ? (n & ~((2u << top) - 1u)) : n;   // common leading bits
    bool done = top < 0, exact = false;
    const int start = __reduce_max_sync(kFullMask, top);
    int bit = start;
    for (; bit >= 16; --bit) {
        if (__all_sync(kFullMask, done)) break;
        const bool act = !done && bit <= top;
        const unsigned cand = thr | (1u << bit);
        const unsigned c2 = (cand >> 16) * 0x00010001u;
        __nv_bfloat162 g[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) g[i] = ge_one_bf16x2(hk[i], c2);
        const __nv_bfloat162 acc = __hadd2(__hadd2(__hadd2(g[0], g[1]), __hadd2(g[2], g[3])),
                                           __hadd2(__hadd2(g[4], g[5]), __hadd2(g[6], g[7])));   // counts <= 8: exact in bf16
        const int cnt = group8_sum(static_cast<int>(__low2float(acc) + __high2float(acc)));
        if (act && cnt >= T) thr = cand;
        if (act && cnt == T) { exact = true; done = true; }
    }
    for (bit = bit > 15 ? 15 : bit; bit >= 0; --bit) {
        if (__all_sync(kFullMask, done)) break;
        const bool act = !done && bit <= top;
        const unsigned cand = thr | (1u << bit);
        int mine = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) mine += (key[i] >= cand) ? 1 : 0;
        const int cnt = group8_sum(mine);
        if (act && cnt >= T) thr = cand;
        if (act && cnt == T) { exact = true; done = true; }
    }
    unsigned kept = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) kept |= (key[i] >= thr) ? (1u << i) : 0u;
    if (__any_sync(kFullMask, !exact)) {
        // not an exact split: thr is the T-th largest key and the keys equal to it are admitted in ascending
        // channel order (lanes ascending, channels inside a lane ascending) until T channels are kept
        int n_gt = 0, n_eq = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            n_gt += (key[i] > thr) ? 1 : 0;
            n_eq += (key[i] == thr) ? 1 : 0;
        }
        const int need_eq = T - group8_sum(n_gt);
        int rank = group8_exclusive(n_eq, l8);
        if (!exact) {
            kept = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const bool eq = key[i] == thr;
                if (key[i] > thr || (eq && rank < need_eq)) kept |= 1u << i;
                rank += eq ? 1 : 0;
            }
        }
    }
    return kept;
}

// One token of one KV head handled by the eight lanes of a group: saliency, selection, and the token's
// entries of the page image.  The lane owns channels 16*l8 .. 16*l8+15; `raw` holds their stored bit patterns
// (two bf16 per word, or one fp32 per word).  Same outputs as pack_token.
template <bool kBf16>
__device__ __forceinline__ void pack_token16(unsigned char* image, int vals_off, int mask_off, int mu_off,
                                             int stats_off, int p, int T, int l8, bool live,
                                             const float* __restrict__ a, const unsigned* raw, double inv_pruned)
{
    unsigned key[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float kf = kBf16 ? __uint_as_float((i & 1) ? (raw[i >> 1] & 0xffff0000u) : (raw[i >> 1] << 16))
                               : __uint_as_float(raw[i]);
        key[i] = __float_as_uint(__fmul_rn(a ? a[i] : 1.f, fabsf(kf)));     // the one rounding that decides selection
    }
    const unsigned kept = select_top_t16(key, T, l8);
    const int slot0 = group8_exclusive(__popc(kept), l8);
    double pruned = 0.0, s1 = 0.0;
    if (live) {
        unsigned char* dst = image + vals_off + val_offset(kBf16 ? 2 : 4, p, slot0);
        constexpr int kRow = kPageTokens * (kBf16 ? 2 : 4);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if ((kept >> i) & 1u) {
                if (kBf16) *reinterpret_cast<unsigned short*>(dst) =
                               static_cast<unsigned short>((i & 1) ? (raw[i >> 1] >> 16) : (raw[i >> 1] & 0xffffu));
                else *reinterpret_cast<unsigned*>(dst) = raw[i];
                dst += kRow;
            } else {
                pruned += static_cast<double>(__uint_as_float(key[i]));
            }
        }
    }
    const unsigned other = __shfl_xor_sync(kFullMask, kept, 1);
    if (live && (l8 & 1) == 0)
        reinterpret_cast<unsigned*>(image + mask_off)[p * kMaskWords + (l8 >> 1)] = kept | (other << 16);
    if (mu_off < 0) return;                                   // warp-uniform
    pruned = group8_sum(pruned);
    if (live && l8 == 0) reinterpret_cast<float*>(image + mu_off)[p] = static_cast<float>(pruned * inv_pruned);
    if (stats_off < 0) return;                                // warp-uniform
#pragma unroll
    for (int i = 0; i < 16; ++i) s1 += static_cast<double>(__uint_as_float(key[i]));
    const double mean = group8_sum(s1) / static_cast<double>(kHeadDim);
    double s2 = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) { const double d = static_cast<double>(__uint_as_float(key[i])) - mean; s2 += d * d; }
    s2 = group8_sum(s2);
    if (live && l8 == 0) {
        reinterpret_cast<float*>(image + stats_off)[p] = static_cast<float>(mean);
        reinterpret_cast<float*>(image + stats_off)[kPageTokens + p] = static_cast<float>(sqrt(s2 / static_cast<double>(kHeadDim)));
    }
}

template <typename E>
__global__ void __launch_bounds__(128, 8) compress_pages4_kernel(CompressArgs A)
{
    grid_wait();
    grid_release();
    extern __shared__ __align__(16) unsigned char image[];
    constexpr bool kBf16 = (sizeof(E) == 2);
    constexpr int kWords = kBf16 ? 8 : 16;                     // 32-bit words of a lane's 16 channels
    const int blk = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int len = A.lens[b];
    if (blk * kPageTokens >= len) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l8 = lane & 7;
    const int p = warp * 4 + (lane >> 3);                      // this group's token of the page
    const PageLayout L = A.L;

    for (int i = threadIdx.x; i < L.page_bytes / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(image)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    float a[16];
    {
        const float4* src = reinterpret_cast<const float4*>(A.qnorm + (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim) + 4 * l8;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 f = src[i];
            a[4 * i] = f.x; a[4 * i + 1] = f.y; a[4 * i + 2] = f.z; a[4 * i + 3] = f.w;
        }
    }
    const int t = blk * kPageTokens + p;
    const bool live = t < len;
    unsigned kraw[kWords], vraw[kWords];
#pragma unroll
    for (int i = 0; i < kWords; ++i) { kraw[i] = 0u; vraw[i] = 0u; }
    if (live) {
        const int src_t = A.gather ? A.gather[(static_cast<int64_t>(b) * A.Hkv + h) * A.gather_stride + t] : t;
        const int64_t row = static_cast<int64_t>(b) * A.sb + static_cast<int64_t>(h) * A.sh +
                            static_cast<int64_t>(src_t) * A.st + l8 * 16;
        const uint4* ks = reinterpret_cast<const uint4*>(static_cast<const E*>(A.k) + row);
        const uint4* vs = reinterpret_cast<const uint4*>(static_cast<const E*>(A.v) + row);
#pragma unroll
        for (int i = 0; i < kWords / 4; ++i) {
            const uint4 kk = ks[i], vv = vs[i];
            kraw[4 * i] = kk.x; kraw[4 * i + 1] = kk.y; kraw[4 * i + 2] = kk.z; kraw[4 * i + 3] = kk.w;
            vraw[4 * i] = vv.x; vraw[4 * i + 1] = vv.y; vraw[4 * i + 2] = vv.z; vraw[4 * i + 3] = vv.w;
        }
        if (L.keep_v >= kHeadDim) {                        // dense value row: the lane's 16-byte chunks
#pragma unroll
            for (int i = 0; i < kWords / 4; ++i)
                *reinterpret_cast<uint4*>(image + L.v_off + v_chunk_offset(kBf16 ? 2 : 4, p, (kWords / 4) * l8 + i)) =
                    make_uint4(vraw[4 * i], vraw[4 * i + 1], vraw[4 * i + 2], vraw[4 * i + 3]);
        }
    }
    if (L.keep_v < kHeadDim)                               // value-channel pruning: same selection on |V|
        pack_token16<kBf16>(image, L.v_off, L.vmask_off, -1, -1, p, L.keep_v, l8, live, nullptr, vraw, 0.0);
    pack_token16<kBf16>(image, L.vals_off, L.mask_off, L.mu_off,
                        L.recovery != SPARK_RECOVER_DEGENERATE ? L.stats_off : -1, p, L.keep, l8, live, a, kraw,
                        A.inv_pruned);
    __syncthreads();

    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    const int64_t page_id = A.block_table ? A.block_table[entry] : entry;     // no table: contiguous cache
    if (page_id < 0 || page_id >= A.n_pool_pages) {
        if (threadIdx.x == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    uint4* dst = reinterpret_cast<uint4*>(A.pages + page_id * L.page_bytes);
    for (int i = threadIdx.x; i < L.page_bytes / 16; i += blockDim.x)
        dst[i] = reinterpret_cast<const uint4*>(image)[i];
}

// ------------------------------------------------------------------------------------------------
// Fixed-T pages of bf16 storage, a page per WARP: a token belongs to two lanes (64 channels each), so a step of the
// selection serves sixteen tokens and needs one shuffle, and a warp owns its page from the loads to the stores
// without a CTA barrier.
//   Selection.  Any threshold t with exactly T keys >= t names the kept set, so the search need not descend bit by bit:
//   it counts over the keys' upper halves, two keys per compare, until T is hit or at most kFewKeys keys lie between the
//   ends; those are ranked against each other by their full bits, in order of key and then of channel.  The first look is at
//   the mean of the token's key bits (the mean of the logarithms, near the median), moved by T's distance from the middle; then
//   by the usual density and a step past the crossing until both ends are known, then false position: 3.8 looks (the most of
//   sixteen tokens, T = 25 .. 89, Gaussian keys) where interpolation from the least and the largest key down to two keys took 8.3.
//   What bounds it: issue slots (168 instructions a token, 71 % of the slots, ALU pipe 58 %), then shared memory (27 wavefronts a token,
//   41 % of its rate).
//   8 heads x 32768 tokens: 104 us with eight lanes per token and a bitwise descent (compress_pages4_kernel, which fp32
//   storage and sampled recovery keep), 60 with the 8.3 looks, 57 now; the same kernel without selection, slots and mean 43.
//   Prefill of 32K tokens, builds in turn: 87.9 -> 86.6 us.  By warps a SM, in one other run: 87.8, 85.7, 95.0, 100.4 with 20, 24, 28, 32.
// ------------------------------------------------------------------------------------------------
constexpr int kWarpPageWarps = 4;      // pages (warps) of a CTA; one where no sequence has more (1000 x 16 tokens: 84 us with four, 57 with one)
constexpr int kFewKeys = 8;            // keys left between the ends that are ranked by their full bits
constexpr int kBitsPerKey = 6;         // steps of the upper half from one key of a token to the next, about (a guess that only costs looks)
constexpr int kAdmitPasses = 4;        // values of the boundary's upper half admitted one by one; more go to the bitwise descent
constexpr int kTileBytes = kPageTokens * kHeadDim * 2;
constexpr int kWarpPageFixed = kTileBytes + kPageTokens * kFewKeys * 4;      // a page's rows and its tokens' candidates

__device__ __forceinline__ unsigned bits_min2(unsigned a, unsigned b)          // bf16 pairs; a NaN loses
{
    const __nv_bfloat162 r = __hmin2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const unsigned*>(&r);
}
__device__ __forceinline__ unsigned ge_mask_bf16x2(unsigned a, unsigned b)     // 0xFFFF per half where a >= b
{
    return __hge2_mask(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
}
// keys of this lane at or above the threshold (its upper half in both halves of t2)
__device__ __forceinline__ int count_ge(const unsigned (&hk)[32], unsigned t2)
{
    __nv_bfloat162 c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = ge_one_bf16x2(hk[i], t2);
#pragma unroll
    for (int j = 4; j < 32; ++j) c[j & 3] = __hadd2(c[j & 3], ge_one_bf16x2(hk[j], t2));   // counts <= 32: exact in bf16
    const __nv_bfloat162 t = __hadd2(__hadd2(c[0], c[1]), __hadd2(c[2], c[3]));
    return static_cast<int>(__low2float(t) + __high2float(t));
}
// full key of channel ch (0..63) of this lane's half row
template <bool kValue>
__device__ __forceinline__ unsigned full_key(const unsigned char* row, int sw, int half, int ch, const float* a)
{
    const int c = 8 * half + (ch >> 3);
    const unsigned short h = *reinterpret_cast<const unsigned short*>(row + ((c ^ sw) << 4) + (ch & 7) * 2);
    const float x = fabsf(bf16_bits_to_float(h));
    return __float_as_uint(kValue ? x : __fmul_rn(a[ch], x));
}

// Mask words of a token from its kept channels 4 * lane .. 4 * lane + 3 (whole warp).
__device__ __forceinline__ uint4 mask_words(const bool (&kept)[4], int lane)
{
    unsigned nib = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) nib |= kept[i] ? (1u << i) : 0u;
    const unsigned w = nib << (4 * (lane & 7));
    uint4 m;
    m.x = __reduce_or_sync(kFullMask, lane < 8 ? w : 0u);
    m.y = __reduce_or_sync(kFullMask, (lane >> 3) == 1 ? w : 0u);
    m.z = __reduce_or_sync(kFullMask, (lane >> 3) == 2 ? w : 0u);
    m.w = __reduce_or_sync(kFullMask, lane >= 24 ? w : 0u);
    return m;
}
// Mask words of one token by the bitwise descent (called by the whole warp, rarely, so out of line).  Keys that nearly all
// share their upper half (constant keys under window means within 1 % of each other) are its case: admitted value by value
// 8192 such tokens took 328 us a prefill (the descent for every token 39), this takes 67.
template <bool kValue>
__device__ __noinline__ uint4 descent_mask(const unsigned char* row, int sw, int lane, int T, const float* a)
{
    const uint2 v = *reinterpret_cast<const uint2*>(row + (((lane >> 1) ^ sw) << 4) + (lane & 1) * 8);
    const float f[4] = {__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u)};
    unsigned key[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) key[i] = __float_as_uint(kValue ? fabsf(f[i]) : __fmul_rn(a[4 * lane + i], fabsf(f[i])));
    bool kept[4];
    select_top_t(key, T, lane, kept);
    return mask_words(kept, lane);
}

// The `need` largest of a token's candidates when more than kFewKeys share one upper half (whole warp, tokens without need
// idle; rare, so out of line): value by value, equal keys in ascending channel order, many distinct ones by the descent.
// Returns the lane's admitted channels (every key above the candidates may be among them).
template <bool kValue>
__device__ __noinline__ unsigned long long admit_many(const unsigned char* tile, unsigned long long cand, int need, int T, int lane, const float* a_all)
{
    const int p = lane & 15, half = lane >> 4, sw = p & 7;
    const unsigned char* row = tile + p * (kHeadDim * 2);
    const float* a = a_all + 64 * half;
    unsigned long long got = 0ull;
    for (int pass = 0; __any_sync(kFullMask, need > 0); ++pass) {
        if (pass == kAdmitPasses || (pass == 1 && __any_sync(kFullMask, need > 0 && __popcll(cand) > 8))) {   // many distinct keys in one upper half
            for (unsigned todo = __ballot_sync(kFullMask, need > 0) & 0xffffu; todo; todo &= todo - 1) {
                const int tok = __ffs(todo) - 1;
                const uint4 m = descent_mask<kValue>(tile + tok * (kHeadDim * 2), tok & 7, lane, T, a_all);
                if (p == tok) got = half ? (static_cast<unsigned long long>(m.w) << 32) | m.z : (static_cast<unsigned long long>(m.y) << 32) | m.x;
            }
            break;
        }
        unsigned best = 0u;                                     // largest full key left (keys compare as their bits)
        unsigned long long eq = 0ull;
        for (unsigned long long m = need > 0 ? cand : 0ull; m; m &= m - 1) {
            const int ch = __ffsll(static_cast<long long>(m)) - 1;
            const unsigned k = full_key<kValue>(row, sw, half, ch, a);
            if (k > best) { best = k; eq = 0ull; }
            if (k == best) eq |= 1ull << ch;
        }
        const unsigned other = __shfl_xor_sync(kFullMask, best, 16);
        if (other > best) eq = 0ull;
        const int mine = __popcll(eq), theirs = __shfl_xor_sync(kFullMask, mine, 16);
        int take = half ? need - theirs : need;                 // equal keys: lower channels first
        take = take < 0 ? 0 : (take > mine ? mine : take);
        unsigned long long rest = eq;
        for (int k = 0; k < take; ++k) rest &= rest - 1;
        got |= eq & ~rest;
        cand &= ~eq;
        need -= mine + theirs;
        if (mine + theirs == 0) need = 0;                       // (no candidate left)
    }
    return got;
}

// One section of a page from the rows in `tile` (16 rows of 256 bytes, 16-byte chunk c of row p at c ^ (p & 7)): kept
// values in slot order, mask words, and for keys (kValue false) the mean of the pruned saliencies.
template <bool kValue>
__device__ __forceinline__ void select_section(const unsigned char* tile, unsigned char* image, int vals_off, int mask_off,
                                               int mu_off, int T, int n, int lane, const float* a_all, double inv_pruned, unsigned* list)
{
    const int p = lane & 15, half = lane >> 4, sw = p & 7;
    const bool live = p < n;
    const unsigned char* row = tile + p * (kHeadDim * 2);
    const float* a = a_all + 64 * half;
    unsigned kept[2] = {live ? 0xffffffffu : 0u, live ? 0xffffffffu : 0u};
    if (T < kHeadDim) {
        // upper halves of the keys: word 16 g + j holds channels 32 g + j (low) and 32 g + 16 + j (high)
        unsigned hk[32];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            unsigned w[16];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 v = *reinterpret_cast<const uint4*>(row + (((8 * half + 4 * g + c) ^ sw) << 4));
                const unsigned x[4] = {v.x, v.y, v.z, v.w};
                if (kValue) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {               // |V| itself is the key
                        const unsigned m = x[j] & 0x7fff7fffu;
                        const int i0 = 8 * c + 2 * j;
                        if (i0 < 16) { w[i0] = m & 0xffffu; w[i0 + 1] = m >> 16; }
                        else { w[i0 - 16] |= m << 16; w[i0 - 15] |= m & 0xffff0000u; }
                    }
                } else {
                    const float4 f0 = *reinterpret_cast<const float4*>(a + 32 * g + 8 * c);
                    const float4 f1 = *reinterpret_cast<const float4*>(a + 32 * g + 8 * c + 4);
                    const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const unsigned k0 = __float_as_uint(__fmul_rn(f[2 * j], fabsf(__uint_as_float(x[j] << 16))));
                        const unsigned k1 = __float_as_uint(__fmul_rn(f[2 * j + 1], fabsf(__uint_as_float(x[j] & 0xffff0000u))));
                        const int i0 = 8 * c + 2 * j;
                        if (i0 < 16) { w[i0] = k0; w[i0 + 1] = k1; }
                        else { w[i0 - 16] = __byte_perm(w[i0 - 16], k0, 0x7632); w[i0 - 15] = __byte_perm(w[i0 - 15], k1, 0x7632); }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) hk[16 * g + j] = w[j];
        }
        // mean of the keys' bits (= of their logarithms), and whether a NaN is among them
        unsigned sum = 0u;
        __nv_bfloat162 nan2 = *reinterpret_cast<const __nv_bfloat162*>(&hk[0]);
#pragma unroll
        for (int j = 0; j < 32; ++j) sum = __dp2a_lo(hk[j], 0x0101u, sum);
#pragma unroll
        for (int j = 1; j < 32; ++j) nan2 = __hadd2(nan2, *reinterpret_cast<const __nv_bfloat162*>(&hk[j]));      // non-negative numbers: NaN only from NaN
        sum += __shfl_xor_sync(kFullMask, sum, 16);
        if (__any_sync(kFullMask, __hisnan(nan2.x) || __hisnan(nan2.y))) {      // NaN saliencies order above infinity, by their bits
#pragma unroll
            for (int j = 0; j < 32; ++j) hk[j] = bits_min2(hk[j], 0x7f807f80u);
        }
        int lo = 0, hi = 0x7f81, c_lo = kHeadDim, c_hi = 0;    // counts at lo (>= T) and hi (< T)
        int t = static_cast<int>(sum >> 7) + (kHeadDim / 2 - T) * kBitsPerKey, c = T, pad = kBitsPerKey, side = 0;
        // weights of the two ends (distances of their counts from T; an end that stays while the other moves twice counts half:
        // the "Illinois" false position), every sixth step bisects
        float w_lo = static_cast<float>(kHeadDim - T) + 0.5f, w_hi = static_cast<float>(T) - 0.5f;
        bool done = !live;
#pragma unroll 1
        for (int it = 0; !__all_sync(kFullMask, done); ++it) {
            const int span = hi - lo;
            if (it % 6 == 5) t = lo + (span >> 1);
            else if (it > 0 && (lo == 0 || hi == 0x7f81)) {    // one end not found yet: by the usual density, and past the crossing
                t += (c - T) * kBitsPerKey + (c > T ? pad : -pad);
                pad = min(2 * pad, 0x4000);
            } else if (it > 0) t = lo + static_cast<int>(static_cast<float>(span) * __fdividef(w_lo, w_lo + w_hi));
            t = max(lo + 1, min(t, hi - 1));
            c = count_ge(hk, static_cast<unsigned>(t) * 0x00010001u);
            c += __shfl_xor_sync(kFullMask, c, 16);
            if (!done) {
                if (c >= T) {
                    lo = t; c_lo = c;
                    w_lo = static_cast<float>(c - T) + 0.5f;
                    if (side > 0) w_hi *= 0.5f;
                    side = 1;
                } else {
                    hi = t; c_hi = c;
                    w_hi = static_cast<float>(T - c) - 0.5f;
                    if (side < 0) w_lo *= 0.5f;
                    side = -1;
                }
                done = c == T || hi - lo == 1 || c_lo - c_hi <= kFewKeys;
            }
        }
        // keys at or above lo; the kept set when there are exactly T of them
        const unsigned t2 = static_cast<unsigned>(lo) * 0x00010001u;
        unsigned ge[2] = {0u, 0u};
#pragma unroll
        for (int j = 0; j < 32; ++j) ge[j >> 4] |= ge_mask_bf16x2(hk[j], t2) & (0x00010001u << (j & 15));
        const int need = live && c_lo != T ? T - c_hi : 0;     // keys between the ends to admit
        kept[0] &= ge[0]; kept[1] &= ge[1];
        if (__any_sync(kFullMask, need > 0)) {
            const unsigned u2 = static_cast<unsigned>(hi) * 0x00010001u;
            unsigned gt[2] = {0u, 0u};
            if (hi <= 0x7f80) {
#pragma unroll
                for (int j = 0; j < 32; ++j) gt[j >> 4] |= ge_mask_bf16x2(hk[j], u2) & (0x00010001u << (j & 15));
            }
            unsigned long long cand = 0ull;
            if (need > 0) cand = (static_cast<unsigned long long>(ge[1] & ~gt[1]) << 32) | (ge[0] & ~gt[0]);
            const bool many = c_lo - c_hi > kFewKeys;
            // up to kFewKeys candidates in channel order, ranked against each other by their full bits
            unsigned* mylist = list + p * kFewKeys;
            *reinterpret_cast<uint4*>(mylist + 4 * half) = make_uint4(0u, 0u, 0u, 0u);
            const int mine = __popcll(cand), theirs = __shfl_xor_sync(kFullMask, mine, 16), first = half ? theirs : 0;
            __syncwarp();
            {
                int i = first;
                for (unsigned long long m = many ? 0ull : cand; m; m &= m - 1, ++i)
                    mylist[i] = full_key<kValue>(row, sw, half, __ffsll(static_cast<long long>(m)) - 1, a);
            }
            __syncwarp();
            const uint4 k0 = *reinterpret_cast<const uint4*>(mylist), k1 = *reinterpret_cast<const uint4*>(mylist + 4);
            const unsigned k[kFewKeys] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
            unsigned admit = 0u;                                // a lane ranks four of them
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const unsigned own = half ? k[4 + e] : k[e], between = half ? own : own + 1u;
                int above = 0;                                  // equal keys: lower channels first
#pragma unroll
                for (int j = 0; j < kFewKeys; ++j) above += k[j] >= (j < e ? own : (j >= 4 + e ? own + 1u : between)) ? 1 : 0;
                admit |= above < need ? 1u << e : 0u;
            }
            admit <<= 4 * half;
            admit |= __shfl_xor_sync(kFullMask, admit, 16);
            unsigned long long out = 0ull;
            {
                int i = first;
                for (unsigned long long m = many ? 0ull : cand; m; m &= m - 1, ++i)
                    if (!((admit >> i) & 1u)) out |= m & (0ull - m);
            }
            if (__any_sync(kFullMask, need > 0 && many)) {
                const unsigned long long got = admit_many<kValue>(tile, cand, need > 0 && many ? need : 0, T, lane, a_all);
                if (need > 0 && many) out = cand & ~got;
            }
            kept[0] &= ~static_cast<unsigned>(out); kept[1] &= ~static_cast<unsigned>(out >> 32);
        }
    }
    const int mine = __popc(kept[0]) + __popc(kept[1]);
    const int theirs = __shfl_xor_sync(kFullMask, mine, 16);
    unsigned char* dst = image + vals_off + val_offset(2, p, half ? theirs : 0);
    double pruned = 0.0;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const unsigned kb = kept[g];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint4 v = *reinterpret_cast<const uint4*>(row + (((8 * half + 4 * g + c) ^ sw) << 4));
            const unsigned x[4] = {v.x, v.y, v.z, v.w};
            float f[8];
            if (!kValue) {
                const float4 f0 = *reinterpret_cast<const float4*>(a + 32 * g + 8 * c);
                const float4 f1 = *reinterpret_cast<const float4*>(a + 32 * g + 8 * c + 4);
                f[0] = f0.x; f[1] = f0.y; f[2] = f0.z; f[3] = f0.w; f[4] = f1.x; f[5] = f1.y; f[6] = f1.z; f[7] = f1.w;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned h = (i & 1) ? x[i >> 1] >> 16 : x[i >> 1] & 0xffffu;
                const bool keep = (kb >> (8 * c + i)) & 1u;
                if (keep) {
                    *reinterpret_cast<unsigned short*>(dst) = static_cast<unsigned short>(h);
                    dst += kPageTokens * 2;
                }
                if (!kValue) pruned += static_cast<double>(keep ? 0.f : __fmul_rn(f[i], fabsf(__uint_as_float(h << 16))));
            }
        }
    }
    *reinterpret_cast<uint2*>(image + mask_off + p * 16 + half * 8) = make_uint2(kept[0], kept[1]);
    if (!kValue) {
        pruned += __shfl_xor_sync(kFullMask, pruned, 16);
        if (half == 0) reinterpret_cast<float*>(image + mu_off)[p] = live ? static_cast<float>(pruned * inv_pruned) : 0.f;
    }
}

template <bool kPV, int kWarps>
__global__ void __launch_bounds__(kWarps * 32, kWarps == 1 ? 1 : (kPV ? 5 : 6)) compress_pages_warp_kernel(CompressArgs A)
{
    extern __shared__ __align__(16) unsigned char page_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = blockIdx.x * kWarps + warp, h = blockIdx.y, b = blockIdx.z;
    const PageLayout L = A.L;
    const int image_bytes = kPV ? L.page_bytes : L.v_off;      // (dense value rows go straight to the page)
    float* a_s = reinterpret_cast<float*>(page_smem);
    unsigned char* tile = page_smem + kHeadDim * 4 + warp * (kWarpPageFixed + image_bytes);
    unsigned* list = reinterpret_cast<unsigned*>(tile + kTileBytes);
    unsigned char* image = tile + kWarpPageFixed;

    // Without eviction the kernel before this one is the window norm, and what it waited for is complete (see
    // grid_release): keys, values and lengths may be read before it ends.
    if (A.gather) { grid_wait(); grid_release(); }
    int len = A.lens[b];
    len = len > A.max_len ? A.max_len : len;
    const int t0 = blk * kPageTokens;
    const int n = len - t0 < kPageTokens ? len - t0 : kPageTokens;
    const int c16 = lane & 15, r2 = lane >> 4;                 // a row per half warp, a 16-byte chunk per lane
    int64_t src_row = t0 + c16;                                 // lane p (p < 16): the source row of token p
    if (A.gather && c16 < n) src_row = A.gather[(static_cast<int64_t>(b) * A.Hkv + h) * A.gather_stride + t0 + c16];
    const int64_t base = static_cast<int64_t>(b) * A.sb + static_cast<int64_t>(h) * A.sh + c16 * 8;
    uint4 kr[8], vr[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int p = 2 * i + r2;
        const int64_t row = base + __shfl_sync(kFullMask, src_row, p) * A.st;
        kr[i] = vr[i] = make_uint4(0, 0, 0, 0);
        if (p < n) {
            kr[i] = *reinterpret_cast<const uint4*>(static_cast<const unsigned short*>(A.k) + row);
            vr[i] = *reinterpret_cast<const uint4*>(static_cast<const unsigned short*>(A.v) + row);
        }
    }
    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    int64_t page_id = 0;
    if (n > 0) page_id = A.block_table ? A.block_table[entry] : entry;        // no table: contiguous cache
    const bool page_ok = page_id >= 0 && page_id < A.n_pool_pages;
    if (!A.gather) { grid_wait(); grid_release(); }
#pragma unroll
    for (int i = 0; i < kHeadDim / (32 * kWarps); ++i)
        a_s[i * (32 * kWarps) + threadIdx.x] = A.qnorm[(static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim + i * (32 * kWarps) + threadIdx.x];
    __syncthreads();
    if (n <= 0) return;                                        // warp-uniform; no CTA barrier below
    if (!page_ok) {
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    unsigned char* page = A.pages + page_id * L.page_bytes;
    if (n < kPageTokens)                                       // slots past the end of the sequence are zero
        for (int i = lane; i < image_bytes / 16; i += 32) reinterpret_cast<uint4*>(image)[i] = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int p = 2 * i + r2, off = p * (kHeadDim * 2) + ((c16 ^ (p & 7)) << 4);
        if (kPV) *reinterpret_cast<uint4*>(tile + off) = vr[i];
        else {
            *reinterpret_cast<uint4*>(page + L.v_off + off) = vr[i];
            *reinterpret_cast<uint4*>(tile + off) = kr[i];
        }
    }
    __syncwarp();
    if (kPV) {                                                 // value-channel pruning: the same selection on |V|
        select_section<true>(tile, image, L.v_off, L.vmask_off, 0, L.keep_v, n, lane, a_s, 0.0, list);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int p = 2 * i + r2;
            *reinterpret_cast<uint4*>(tile + p * (kHeadDim * 2) + ((c16 ^ (p & 7)) << 4)) = kr[i];
        }
        __syncwarp();
    }
    select_section<false>(tile, image, L.vals_off, L.mask_off, L.mu_off, L.keep, n, lane, a_s, A.inv_pruned, list);
    __syncwarp();
    for (int i = lane; i < image_bytes / 16; i += 32)
        reinterpret_cast<uint4*>(page)[i] = reinterpret_cast<const uint4*>(image)[i];
}

// ------------------------------------------------------------------------------------------------
// SparK-p pages of bf16 storage with dense values: per token the fewest most salient channels whose saliencies (summed in
// double) reach top_p of the token's total, at least one and at most T.  Half a page per warp: a token belongs to four
// lanes (channels 32 q .. 32 q + 31 = mask word q), which hold its saliencies in registers.
//   A threshold on the keys' upper halves is searched by the sum R of the keys BELOW it, in fp32, against what the rule
//   leaves out (total - goal), until fewer than kFewBelow keys can lie between the ends.  log R is nearly linear in the key's
//   bits (= log2 of the key), so a first look, a secant and one step past the crossing usually leave two or three looks
//   more: 4.7 looks (the most of eight tokens) for p = 0.5 .. 0.99 on Gaussian keys, where bisections and interpolation of
//   the sum above took 11.  The sum below the lower end is then taken in double, and the keys between are ranked against
//   each other.
//   The rank sort of the append kernels (rank_mask, 2100 instructions a token) still decides where this could decide
//   otherwise: a total that is not finite, a sum within rounding of the goal whose terms do not add up exactly, ends that fp32
//   had put wrong, many keys with one upper half.
//   What bounds it: latency (fixed and of shared memory) more than issue slots, hence as many warps as 64 registers allow: us
//   per prefill of 8192 tokens, p = 0.99, with 20, 24, 28, 32, 36, 40 warps a SM 49.8, 51.5, 52.0, 47.0, 47.0, 51.9.  Two
//   lanes per token with the saliencies in shared memory and 16 warps a SM took 62.3 (8192 tokens), 102.5 (16000 tokens, now
//   70.5), 28.3 (500 tokens, p = 0.95, now 22.2).
// ------------------------------------------------------------------------------------------------
constexpr int kToppWarps = 4;          // two pages a CTA; one (two warps) where no sequence has more
constexpr int kFewBelow = 8;           // keys between the ends that are ranked against each other
constexpr int kToppStride = 36;        // floats between the four lanes' window norms (32 + 4: different banks)
// shared memory of a page: its keys | the candidates of its tokens | rows used of the two halves | mask | mu | slot rows
constexpr int kToppImage = kTileBytes + kPageTokens * kFewBelow * 4 + 16;
__host__ __device__ inline int topp_page_room(const PageLayout& L) { return kToppImage + L.v_off + L.keep * kPageTokens * 2; }

__device__ __forceinline__ int topp_chunk(int c, int row) { return ((c ^ ((c >> 3) << 1)) ^ (row & 7)) << 4; }    // 16-byte chunk c of a row: conflict-free by rows and by lanes
template <typename N> __device__ __forceinline__ N quad_sum(N v)
{
    v += __shfl_xor_sync(kFullMask, v, 1);
    v += __shfl_xor_sync(kFullMask, v, 2);
    return v;
}
__device__ __forceinline__ int quad_exclusive(int v, int q)                // sum over the lower lanes of the four
{
    int x = v, t = __shfl_up_sync(kFullMask, x, 1, 4);
    if (q >= 1) x += t;
    t = __shfl_up_sync(kFullMask, x, 2, 4);
    if (q >= 2) x += t;
    return x - v;
}
__device__ __forceinline__ void pair_sync(int pg)                          // the two warps of a page
{
    if (pg == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
    else asm volatile("bar.sync 2, 64;" ::: "memory");
}

// Mask words of one token by the rank sort that the append kernels use (whole warp; rarely needed, so out of line).
__device__ __noinline__ uint4 rank_mask(const unsigned char* row, int tok, int lane, const float* a_s, float top_p, int cap)
{
    const uint2 v = *reinterpret_cast<const uint2*>(row + topp_chunk(lane >> 1, tok) + (lane & 1) * 8);
    const float f[4] = {__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u)};
    const float* a = a_s + (lane >> 3) * kToppStride + 4 * (lane & 7);
    unsigned key[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) key[i] = __float_as_uint(__fmul_rn(a[i], fabsf(f[i])));
    SelectArgs sel;
    sel.select = SPARK_SELECT_TOP_P; sel.top_p = top_p; sel.recovery = SPARK_RECOVER_DEGENERATE;
    sel.rank_keep[0] = sel.rank_keep[1] = sel.rank_keep[2] = sel.rank_keep[3] = 0u;
    bool kept[4];
    select_by_rank(key, lane, sel, cap, kept);
    return mask_words(kept, lane);
}

// What the search leaves open (whole warp; rare, so out of line): tokens whose sums decide only if they add up exactly
// (`near`), tokens for the rank sort, tokens over the page's capacity (by `drop`), and sums to be taken again.
__device__ __noinline__ unsigned topp_settle(const unsigned char* tile, int T, float top_p, bool near, bool rank, int drop,
                                             unsigned got, int lane, const float* a_s, double& pruned)
{
    const int p8 = lane >> 2, q = lane & 3;
    const unsigned char* row = tile + p8 * (kHeadDim * 2);
    const float* a = a_s + q * kToppStride;
    auto sal = [&](int r) {
        const unsigned short x = *reinterpret_cast<const unsigned short*>(row + topp_chunk(4 * q + (r >> 3), p8) + (r & 7) * 2);
        return __fmul_rn(a[r], fabsf(bf16_bits_to_float(x)));
    };
    if (__any_sync(kFullMask, near)) {
        // 128 terms add up exactly in double, in any order, when their exponents span at most 22
        unsigned least = 0x7f800000u, most = 0u;
#pragma unroll 4
        for (int r = 0; r < 32; ++r) {
            const unsigned x = __float_as_uint(sal(r));
            least = x ? min(least, x) : least;
            most = max(most, x);
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            least = min(least, __shfl_xor_sync(kFullMask, least, o));
            most = max(most, __shfl_xor_sync(kFullMask, most, o));
        }
        rank = rank || (near && static_cast<int>(most >> 23) - static_cast<int>(least >> 23) > 22);
    }
    unsigned flags = __ballot_sync(kFullMask, rank);           // any lane of a token
    flags |= flags >> 1; flags |= flags >> 2;
    for (unsigned todo = flags & 0x11111111u; todo; todo &= todo - 1) {
        const int tok = (__ffs(todo) - 1) >> 2;
        const uint4 m = rank_mask(tile + tok * (kHeadDim * 2), tok, lane, a_s, top_p, T);
        if (p8 == tok) { got = q & 2 ? (q & 1 ? m.w : m.z) : (q & 1 ? m.y : m.x); drop = 0; }
    }
    // drop the least salient, higher channels first, until T are left
    for (; __any_sync(kFullMask, drop > 0); --drop) {
        unsigned low = 0xffffffffu;
        int at = -1;
        for (unsigned m = drop > 0 ? got : 0u; m; m &= m - 1) {
            const int r = __ffs(m) - 1;
            const unsigned x = __float_as_uint(sal(r));
            if (x <= low) { low = x; at = 32 * q + r; }
        }
        int best = at;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const unsigned other = __shfl_xor_sync(kFullMask, low, o);
            const int other_at = __shfl_xor_sync(kFullMask, best, o);
            if (other < low || (other == low && other_at > best)) { low = other; best = other_at; }
        }
        if (drop > 0 && best == at && at >= 0) got &= ~(1u << (at & 31));
    }
    double s = 0.0;
#pragma unroll 4
    for (int r = 0; r < 32; ++r)
        if (!((got >> r) & 1u)) s += static_cast<double>(sal(r));
    pruned = quad_sum(s);
    return got;
}

// Kept channels of this lane (bit r: channel 32 q + r) of the eight tokens whose key rows lie in `tile`; `pruned` receives
// the token's sum of the others.  `list`: room for the tokens' candidates.
__device__ __forceinline__ unsigned select_topp(const unsigned char* tile, float* list, int T, float top_p, bool live, int lane,
                                                const float* a_s, double& pruned)
{
    const int p8 = lane >> 2, q = lane & 3;
    const unsigned char* row = tile + p8 * (kHeadDim * 2);
    const float* a = a_s + q * kToppStride;
    list += p8 * kFewBelow;
    float w[32], top_w = 0.f;
    double t0 = 0.0, t1 = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint4 v = *reinterpret_cast<const uint4*>(row + topp_chunk(4 * q + c, p8));
        const unsigned x[4] = {v.x, v.y, v.z, v.w};
        const float4 f0 = *reinterpret_cast<const float4*>(a + 8 * c), f1 = *reinterpret_cast<const float4*>(a + 8 * c + 4);
        const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float x0 = __fmul_rn(f[2 * j], fabsf(__uint_as_float(x[j] << 16)));      // the one rounding that decides selection
            const float x1 = __fmul_rn(f[2 * j + 1], fabsf(__uint_as_float(x[j] & 0xffff0000u)));
            w[8 * c + 2 * j] = x0; w[8 * c + 2 * j + 1] = x1;
            top_w = fmaxf(top_w, fmaxf(x0, x1));
            t0 += static_cast<double>(x0);
            t1 += static_cast<double>(x1);
        }
    }
    top_w = fmaxf(top_w, __shfl_xor_sync(kFullMask, top_w, 1));
    top_w = fmaxf(top_w, __shfl_xor_sync(kFullMask, top_w, 2));
    const double total = quad_sum(t0 + t1), goal = static_cast<double>(top_p) * total, left = total - goal;
    const bool finite = total < static_cast<double>(INFINITY);                  // (false for NaN)
    const bool search = live && finite && top_w > 0.f;
    const float left_f = static_cast<float>(left), log_left = __log2f(left_f);
    // ends of the search (upper halves): the keys below l sum up to what may be left out, those below h to more
    const int h0 = static_cast<int>(__float_as_uint(top_w) >> 16) + 1;
    int l = 0, h = h0, t = 0, pad = 14, side = 0;
    float r_l = 0.f, r_h = static_cast<float>(total), y = 0.f, y_l = -INFINITY, y_h = __log2f(r_h) - log_left;     // y: log2(R / left)
    bool done = !search;
#pragma unroll 1
    for (int it = 0;; ++it) {
        const int span = h - l;
        const float v_l = __uint_as_float(static_cast<unsigned>(l) << 16);
        if (span <= 1 || (l > 0 && r_h - r_l < (kFewBelow - 0.1f) * v_l)) done = true;     // every key between the ends is at least v_l
        if (__all_sync(kFullMask, done)) break;
        if (it == 0) t = static_cast<int>(__float_as_uint(left_f * 0.05f) >> 16);            // some forty keys of half the threshold's size
        else if (it % 5 == 4 || !(left_f > 0.f)) t = l + (span >> 1);
        else if (l == 0 || h == h0) {                          // one end not found yet: along R ~ t^1.4, and past the crossing
            t += static_cast<int>(fminf(fmaxf(-y, -3.f), 3.f) * 91.f) + (y <= 0.f ? pad : -pad);
            pad = min(2 * pad, 4096);
        } else if (!(y_l > -INFINITY)) t = h - static_cast<int>(y_h * 91.f) - 14;
        else t = l + static_cast<int>(static_cast<float>(span) * __fdividef(-y_l, y_h - y_l));
        t = max(l + 1, min(t, h - 1));
        const float tf = __uint_as_float(static_cast<unsigned>(t) << 16);
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int r = 0; r < 32; ++r)
            if (w[r] < tf) s[r & 3] += w[r];
        const float below = quad_sum((s[0] + s[1]) + (s[2] + s[3]));
        if (!done) {
            y = below > 0.f ? __log2f(below) - log_left : -INFINITY;
            if (below <= left_f) { l = t; r_l = below; y_l = y; if (side > 0) y_h *= 0.5f; side = 1; }
            else { h = t; r_h = below; y_h = y; if (side < 0) y_l *= 0.5f; side = -1; }
        }
    }
    const float lo = __uint_as_float(static_cast<unsigned>(l) << 16), hi = __uint_as_float(static_cast<unsigned>(h) << 16);
    unsigned got = 0u, cand = 0u;                              // keys >= hi; keys in [lo, hi)
    t0 = t1 = 0.0;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const bool ge = w[r] >= lo;
        got |= w[r] >= hi ? 1u << r : 0u;
        cand |= ge ? 1u << r : 0u;
        (r & 1 ? t1 : t0) += static_cast<double>(ge ? 0.f : w[r]);
    }
    cand &= ~got;
    pruned = t0 + t1;
    if (!search) { got = live && top_w == 0.f && q == 0 ? 1u : 0u; cand = 0u; }            // all saliencies zero: the first channel
    // candidates in channel order
    const int mine = __popc(cand), first = quad_exclusive(mine, q), nc = quad_sum(mine), na = quad_sum(__popc(got));
    {
        int i = first;
        for (unsigned m = cand; m; m &= m - 1, ++i) {
            const int r = __ffs(m) - 1;
            const unsigned short x = *reinterpret_cast<const unsigned short*>(row + topp_chunk(4 * q + (r >> 3), p8) + (r & 7) * 2);
            if (i < kFewBelow) list[i] = __fmul_rn(a[r], fabsf(bf16_bits_to_float(x)));
        }
    }
    __syncwarp();
    float k[kFewBelow];
    {
        const float4 k0 = *reinterpret_cast<const float4*>(list), k1 = *reinterpret_cast<const float4*>(list + 4);
        k[0] = k0.x; k[1] = k0.y; k[2] = k0.z; k[3] = k0.w; k[4] = k1.x; k[5] = k1.y; k[6] = k1.z; k[7] = k1.w;
    }
    double between = 0.0;
#pragma unroll
    for (int i = 0; i < kFewBelow; ++i) if (i < nc) between += static_cast<double>(k[i]);
    const double reach = total - quad_sum(pruned);             // the keys >= lo
    const double above = na > 0 ? reach - between : 0.0;       // the keys >= hi
    const double slack = total * 0x1p-44;                      // more than 128 roundings
    bool near = fabs(reach - goal) <= slack || fabs(above - goal) <= slack;
    unsigned admit = 0u;                                       // a lane decides on two candidates: admitted when the sum before falls short
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = 2 * q + e;
        const float own = e ? (q & 2 ? (q & 1 ? k[7] : k[5]) : (q & 1 ? k[3] : k[1])) : (q & 2 ? (q & 1 ? k[6] : k[4]) : (q & 1 ? k[2] : k[0]));
        double before = above;
#pragma unroll
        for (int j = 0; j < kFewBelow; ++j)
            if (j < nc && (k[j] > own || (k[j] == own && j < i))) before += static_cast<double>(k[j]);      // equal keys: lower channels first
        if (i < nc) {
            near = near || fabs(before - goal) <= slack;
            if (before < goal) admit |= 1u << i;
        }
    }
    admit |= __shfl_xor_sync(kFullMask, admit, 1);
    admit |= __shfl_xor_sync(kFullMask, admit, 2);
    {
        int i = first;
        for (unsigned m = nc <= kFewBelow ? cand : 0u; m; m &= m - 1, ++i) {
            if ((admit >> i) & 1u) got |= m & (0u - m);
            else pruned += static_cast<double>(list[i]);
        }
    }
    const bool rank = live && (!finite || (search && (nc > kFewBelow || (na > 0 && above >= goal) || reach < goal)));
    const int drop = quad_sum(__popc(got)) - T;                // over the page's capacity
    near = near && search;
    if (__any_sync(kFullMask, (live && !search) || near || rank || drop > 0))
        return topp_settle(tile, T, top_p, near, rank, drop, got, lane, a_s, pruned);
    pruned = quad_sum(pruned);
    return got;
}

template <int kWarps>
__global__ void __launch_bounds__(kWarps * 32, kWarps == 2 ? 1 : 8) compress_topp_kernel(CompressArgs A)
{
    extern __shared__ __align__(16) unsigned char topp_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, pg = warp >> 1, hw = warp & 1;
    const int blk = blockIdx.x * (kWarps / 2) + pg, h = blockIdx.y, b = blockIdx.z;
    const PageLayout L = A.L;
    float* a_s = reinterpret_cast<float*>(topp_smem);
    unsigned char* own = topp_smem + 4 * kToppStride * 4 + pg * topp_page_room(L);
    unsigned char* tile = own + hw * (kTileBytes / 2);
    float* list = reinterpret_cast<float*>(own + kTileBytes) + hw * 8 * kFewBelow;
    int* rows_used = reinterpret_cast<int*>(own + kTileBytes + kPageTokens * kFewBelow * 4);
    unsigned char* image = own + kToppImage;

    if (A.gather) { grid_wait(); grid_release(); }             // what may be read before: as in compress_pages_warp_kernel
    int len = A.lens[b];
    len = len > A.max_len ? A.max_len : len;
    const int t0 = blk * kPageTokens;
    const int n = len - t0 < kPageTokens ? len - t0 : kPageTokens;
    const int c16 = lane & 15, r2 = lane >> 4;                 // a row per half warp, a 16-byte chunk per lane
    int64_t src_row = t0 + 8 * hw + (lane & 7);
    if (A.gather && 8 * hw + (lane & 7) < n) src_row = A.gather[(static_cast<int64_t>(b) * A.Hkv + h) * A.gather_stride + src_row];
    const int64_t base = static_cast<int64_t>(b) * A.sb + static_cast<int64_t>(h) * A.sh + c16 * 8;
    uint4 kr[4], vr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t row = base + __shfl_sync(kFullMask, src_row, 2 * i + r2) * A.st;
        kr[i] = vr[i] = make_uint4(0, 0, 0, 0);
        if (8 * hw + 2 * i + r2 < n) {
            kr[i] = *reinterpret_cast<const uint4*>(static_cast<const unsigned short*>(A.k) + row);
            vr[i] = *reinterpret_cast<const uint4*>(static_cast<const unsigned short*>(A.v) + row);
        }
    }
    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    int64_t page_id = 0;
    if (n > 0) page_id = A.block_table ? A.block_table[entry] : entry;        // no table: contiguous cache
    const bool page_ok = page_id >= 0 && page_id < A.n_pool_pages;
    for (int i = (hw << 5) + lane; i < L.keep * 2; i += 64) reinterpret_cast<uint4*>(image + L.v_off)[i] = make_uint4(0, 0, 0, 0);
    if (!A.gather) { grid_wait(); grid_release(); }
#pragma unroll
    for (int j = threadIdx.x; j < kHeadDim; j += kWarps * 32)
        a_s[(j >> 5) * kToppStride + (j & 31)] = A.qnorm[(static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim + j];
    __syncthreads();                                           // (the cleared slot rows too)
    if (n <= 0) return;                                        // both warps of the page; no CTA barrier below
    if (!page_ok) {
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    unsigned char* page = A.pages + page_id * L.page_bytes;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = 2 * i + r2;
        *reinterpret_cast<uint4*>(page + L.v_off + v_chunk_offset(2, 8 * hw + row, c16)) = vr[i];
        *reinterpret_cast<uint4*>(tile + row * (kHeadDim * 2) + topp_chunk(c16, row)) = kr[i];
    }
    __syncwarp();
    const int p8 = lane >> 2, q = lane & 3, p = 8 * hw + p8;
    const bool live = p < n;
    double pruned;
    const unsigned got = select_topp(tile, list, L.keep, A.sel.top_p, live, lane, a_s, pruned);
    const int mine = __popc(got), count = quad_sum(mine);
    unsigned char* dst = image + L.v_off + val_offset(2, p, quad_exclusive(mine, q));
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint4 v = *reinterpret_cast<const uint4*>(tile + p8 * (kHeadDim * 2) + topp_chunk(4 * q + c, p8));
        const unsigned x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if ((got >> (8 * c + i)) & 1u) {
                *reinterpret_cast<unsigned short*>(dst) = static_cast<unsigned short>((i & 1) ? x[i >> 1] >> 16 : x[i >> 1] & 0xffffu);
                dst += kPageTokens * 2;
            }
    }
    reinterpret_cast<unsigned*>(image + L.mask_off)[p * kMaskWords + q] = got;
    if (q == 0)
        reinterpret_cast<float*>(image + L.mu_off)[p] =
            live && count < kHeadDim ? static_cast<float>(pruned / static_cast<double>(kHeadDim - count)) : 0.f;
    const int rows = __reduce_max_sync(kFullMask, count);
    if (lane == 0) rows_used[hw] = rows;
    pair_sync(pg);
    for (int i = (hw << 5) + lane; i < L.v_off / 16 + L.keep * 2; i += 64) {
        unsigned char* to = page + (i < L.v_off / 16 ? i * 16 : L.vals_off + (i - L.v_off / 16) * 16);
        *reinterpret_cast<uint4*>(to) = reinterpret_cast<const uint4*>(image)[i];
    }
    if (hw == 0 && lane == 0) reinterpret_cast<int*>(A.pages + rows_offset(A.n_pool_pages, L.page_bytes))[page_id] = max(rows_used[0], rows_used[1]);
}

// ------------------------------------------------------------------------------------------------
// Decode-time append: one new token per sequence is pruned with the sequence's prefill statistics
// (qnorm) and written into the next token slot of its last page (a fresh page is zeroed first).
// One warp per (sequence, KV head).  With more than 32 KV heads: a CTA per warp, and a second
// one-thread-per-sequence kernel advances packed_lens; otherwise one launch does both (below).
// ------------------------------------------------------------------------------------------------
struct AppendArgs {
    const void* k_new;
    const void* v_new;
    unsigned char* pages;
    const int32_t* block_table;
    int max_blocks;
    int B, Hkv, keep;
    int64_t n_pool_pages;
    PageLayout L;
    const float* qnorm;
    int32_t* packed_lens;
    double inv_pruned;            // 1 / (D - T), 0 when T = D
    SelectArgs sel;
    int* status;
};

template <typename E, bool kRank>
__global__ void __launch_bounds__(32) append_token_kernel(AppendArgs A)
{
    grid_wait();
    grid_release();
    constexpr bool kBf16 = (sizeof(E) == 2);
    const int h = blockIdx.x, b = blockIdx.y, lane = threadIdx.x;
    const PageLayout L = A.L;
    const int t = A.packed_lens[b];
    const int blk = t / kPageTokens, p = t - blk * kPageTokens;
    if (t < 0 || blk >= A.max_blocks) {                       // no room: recorded, nothing written
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    const int64_t page_id = A.block_table ? A.block_table[entry] : entry;
    if (page_id < 0 || page_id >= A.n_pool_pages) {
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    unsigned char* page = A.pages + page_id * L.page_bytes;
    int* rows = L.ragged ? reinterpret_cast<int*>(A.pages + rows_offset(A.n_pool_pages, L.page_bytes)) + page_id : nullptr;
    if (p == 0) {                                             // first token of a page: clear it
        for (int i = lane; i < L.page_bytes / 16; i += 32) reinterpret_cast<uint4*>(page)[i] = make_uint4(0, 0, 0, 0);
        if (rows && lane == 0) *rows = 0;
        __syncwarp();
    }
    const float4 a4 = reinterpret_cast<const float4*>(A.qnorm + (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim)[lane];
    const float a[4] = {a4.x, a4.y, a4.z, a4.w};
    const int64_t row = (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim + lane * 4;
    const int n_kept = pack_token_kv<kBf16, kRank>(page, L, p, lane, a, A.k_new, A.v_new, row, A.inv_pruned, A.sel);
    if (rows && lane == 0) atomicMax(rows, n_kept);
}

// The same for up to 32 KV heads in ONE launch: a CTA per sequence, a warp per KV head.  Every warp reads the
// sequence's length before the first barrier and thread 0 advances it after the second, so no warp can see
// the advanced length.
template <typename E, bool kRank>
__global__ void __launch_bounds__(1024) append_token_cta_kernel(AppendArgs A)
{
    grid_wait();
    grid_release();
    constexpr bool kBf16 = (sizeof(E) == 2);
    const int b = blockIdx.x, h = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const PageLayout L = A.L;
    // ask for the head's rows before the length is known: one round trip less in the chain
    {
        const int64_t unit = static_cast<int64_t>(b) * A.Hkv + h, row = unit * kHeadDim + lane * 4;
        asm volatile("prefetch.global.L1 [%0];" ::"l"(static_cast<const E*>(A.k_new) + row));
        asm volatile("prefetch.global.L1 [%0];" ::"l"(static_cast<const E*>(A.v_new) + row));
        asm volatile("prefetch.global.L1 [%0];" ::"l"(A.qnorm + row));
    }
    const int t = A.packed_lens[b];
    __syncthreads();
    const int blk = t / kPageTokens, p = t - blk * kPageTokens;
    const bool room = t >= 0 && blk < A.max_blocks;
    if (!room) {                                               // no room: recorded, nothing written
        if (threadIdx.x == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
    } else {
        const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
        const int64_t page_id = A.block_table ? A.block_table[entry] : entry;
        if (page_id < 0 || page_id >= A.n_pool_pages) {
            if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        } else {
            unsigned char* page = A.pages + page_id * L.page_bytes;
            int* rows = L.ragged ? reinterpret_cast<int*>(A.pages + rows_offset(A.n_pool_pages, L.page_bytes)) + page_id : nullptr;
            if (p == 0) {                                      // first token of a page: clear it
                for (int i = lane; i < L.page_bytes / 16; i += 32) reinterpret_cast<uint4*>(page)[i] = make_uint4(0, 0, 0, 0);
                if (rows && lane == 0) *rows = 0;
                __syncwarp();
            }
            const float4 a4 = reinterpret_cast<const float4*>(A.qnorm + (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim)[lane];
            const float a[4] = {a4.x, a4.y, a4.z, a4.w};
            const int64_t row = (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim + lane * 4;
            const int n_kept = pack_token_kv<kBf16, kRank>(page, L, p, lane, a, A.k_new, A.v_new, row, A.inv_pruned, A.sel);
            if (rows && lane == 0) atomicMax(rows, n_kept);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && room) A.packed_lens[b] = t + 1;
}

__global__ void append_advance_kernel(AppendArgs A)
{
    grid_wait();
    grid_release();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= A.B) return;
    const int t = A.packed_lens[b];
    if (t >= 0 && t / kPageTokens < A.max_blocks) A.packed_lens[b] = t + 1;
}

// Block append: n_new tokens per sequence at once (the keys a caller has kept dense for a while and now hands
// over for pruning).  Three launches: fresh pages are zeroed, every (sequence, head, new token) gets a warp that
// prunes it exactly like append_token_kernel, packed_lens advances by the tokens that found room.  Up to eight warps a
// CTA: with one, 128 sequences x 8 heads x 64 tokens (65536 CTAs) were bound by starting CTAs, 78 us a call against 53.
struct AppendBlockArgs {
    AppendArgs a;
    int n_new, n_fresh;           // new tokens; pages that can start inside them
};
constexpr int kBlockWarps = 8;

__global__ void __launch_bounds__(kBlockWarps * 32) append_block_clear_kernel(AppendBlockArgs B_)
{
    grid_wait();
    grid_release();
    const AppendArgs& A = B_.a;
    const int h = blockIdx.x, b = blockIdx.y, lane = threadIdx.x & 31, fresh = (blockIdx.z * blockDim.x + threadIdx.x) >> 5;
    const int t0 = A.packed_lens[b];
    if (t0 < 0 || fresh >= B_.n_fresh) return;
    const int blk = (t0 + kPageTokens - 1) / kPageTokens + fresh;          // pages that start at or after t0
    if (static_cast<int64_t>(blk) * kPageTokens >= static_cast<int64_t>(t0) + B_.n_new || blk >= A.max_blocks) return;
    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    const int64_t page_id = A.block_table ? A.block_table[entry] : entry;
    if (page_id < 0 || page_id >= A.n_pool_pages) {
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    uint4* page = reinterpret_cast<uint4*>(A.pages + page_id * A.L.page_bytes);
    for (int i = lane; i < A.L.page_bytes / 16; i += 32) page[i] = make_uint4(0, 0, 0, 0);
    if (A.L.ragged && lane == 0)
        reinterpret_cast<int*>(A.pages + rows_offset(A.n_pool_pages, A.L.page_bytes))[page_id] = 0;
}

template <typename E, bool kRank>
__global__ void __launch_bounds__(kBlockWarps * 32) append_block_token_kernel(AppendBlockArgs B_)
{
    grid_wait();
    grid_release();
    constexpr bool kBf16 = (sizeof(E) == 2);
    const AppendArgs& A = B_.a;
    const int h = blockIdx.x, b = blockIdx.y, tok = (blockIdx.z * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (tok >= B_.n_new) return;
    const PageLayout L = A.L;
    const int t0 = A.packed_lens[b];
    const int64_t t = static_cast<int64_t>(t0) + tok;
    const int64_t blk = t / kPageTokens;
    const int p = static_cast<int>(t - blk * kPageTokens);
    if (t0 < 0 || blk >= A.max_blocks) {                      // no room: recorded, nothing written
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    const int64_t entry = (static_cast<int64_t>(b) * A.Hkv + h) * A.max_blocks + blk;
    const int64_t page_id = A.block_table ? A.block_table[entry] : entry;
    if (page_id < 0 || page_id >= A.n_pool_pages) {
        if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        return;
    }
    unsigned char* page = A.pages + page_id * L.page_bytes;
    const float4 a4 = reinterpret_cast<const float4*>(A.qnorm + (static_cast<int64_t>(b) * A.Hkv + h) * kHeadDim)[lane];
    const float a[4] = {a4.x, a4.y, a4.z, a4.w};
    const int64_t row = ((static_cast<int64_t>(b) * A.Hkv + h) * B_.n_new + tok) * kHeadDim + lane * 4;
    const int n_kept = pack_token_kv<kBf16, kRank>(page, L, p, lane, a, A.k_new, A.v_new, row, A.inv_pruned, A.sel);
    if (L.ragged && lane == 0)
        atomicMax(reinterpret_cast<int*>(A.pages + rows_offset(A.n_pool_pages, L.page_bytes)) + page_id, n_kept);
}

__global__ void append_block_advance_kernel(AppendBlockArgs B_)
{
    grid_wait();
    grid_release();
    const AppendArgs& A = B_.a;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= A.B) return;
    const int t = A.packed_lens[b];
    if (t < 0) return;
    const int64_t room = static_cast<int64_t>(A.max_blocks) * kPageTokens;
    const int64_t want = static_cast<int64_t>(t) + B_.n_new;
    A.packed_lens[b] = static_cast<int>(want < room ? want : (t > room ? t : room));
}

// selection arguments of a parameter block (the rank mask of SparK-g is laid out on the host)
static SelectArgs make_select(const spark_params& p)
{
    SelectArgs s;
    s.select = p.select; s.top_p = p.top_p; s.recovery = p.recovery;
    s.rank_keep[0] = s.rank_keep[1] = s.rank_keep[2] = s.rank_keep[3] = 0u;
    if (p.select == SPARK_SELECT_GROUPS) {
        int start = 0;
        for (int i = 0; i < p.n_groups; ++i) {
            const int size = kHeadDim / p.n_groups + (i < kHeadDim % p.n_groups ? 1 : 0);
            const int kp = group_keep(size, 1, &p.group_prune[i]);          // floor((1 - prune) * size)
            for (int r = start; r < start + kp; ++r) s.rank_keep[r >> 5] |= 1u << (r & 31);
            start += size;
        }
    }
    return s;
}

spark_status launch_append(const spark_params& p, const void* k_new, const void* v_new, void* pages,
                           const int32_t* block_table, int32_t max_blocks, const float* qnorm,
                           int32_t* packed_lens, void* workspace, cudaStream_t stream, int* launches)
{
    AppendArgs A;
    A.k_new = k_new; A.v_new = v_new; A.pages = static_cast<unsigned char*>(pages); A.block_table = block_table;
    A.max_blocks = max_blocks; A.B = p.batch; A.Hkv = p.n_kv_heads; A.keep = p.keep; A.n_pool_pages = p.n_pool_pages;
    A.L = make_layout(p); A.qnorm = qnorm; A.packed_lens = packed_lens;
    A.inv_pruned = p.keep < kHeadDim ? 1.0 / static_cast<double>(kHeadDim - p.keep) : 0.0;
    A.sel = make_select(p);
    A.status = static_cast<int*>(workspace);
    const bool rank = p.select != SPARK_SELECT_FIXED;
    if (p.n_kv_heads <= 32) {                                  // one launch: a CTA per sequence, a warp per KV head
        const int threads = p.n_kv_heads * 32;
        if (p.dtype == SPARK_BF16) {
            if (rank) launch_kernel(append_token_cta_kernel<__nv_bfloat16, true>, dim3(p.batch), dim3(threads), 0, stream, A);
            else launch_kernel(append_token_cta_kernel<__nv_bfloat16, false>, dim3(p.batch), dim3(threads), 0, stream, A);
        } else {
            if (rank) launch_kernel(append_token_cta_kernel<float, true>, dim3(p.batch), dim3(threads), 0, stream, A);
            else launch_kernel(append_token_cta_kernel<float, false>, dim3(p.batch), dim3(threads), 0, stream, A);
        }
        *launches += 1;
        return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
    }
    const dim3 grid(p.n_kv_heads, p.batch);
    if (p.dtype == SPARK_BF16) {
        if (rank) launch_kernel(append_token_kernel<__nv_bfloat16, true>, grid, dim3(32), 0, stream, A);
        else launch_kernel(append_token_kernel<__nv_bfloat16, false>, grid, dim3(32), 0, stream, A);
    } else {
        if (rank) launch_kernel(append_token_kernel<float, true>, grid, dim3(32), 0, stream, A);
        else launch_kernel(append_token_kernel<float, false>, grid, dim3(32), 0, stream, A);
    }
    launch_kernel(append_advance_kernel, dim3((p.batch + 127) / 128), dim3(128), 0, stream, A);
    *launches += 2;
    return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

spark_status launch_append_block(const spark_params& p, const void* k_new, const void* v_new, int32_t n_new,
                                 void* pages, const int32_t* block_table, int32_t max_blocks, const float* qnorm,
                                 int32_t* packed_lens, void* workspace, cudaStream_t stream, int* launches)
{
    if (n_new == 0) return SPARK_OK;
    AppendBlockArgs Bk;
    AppendArgs& A = Bk.a;
    A.k_new = k_new; A.v_new = v_new; A.pages = static_cast<unsigned char*>(pages); A.block_table = block_table;
    A.max_blocks = max_blocks; A.B = p.batch; A.Hkv = p.n_kv_heads; A.keep = p.keep; A.n_pool_pages = p.n_pool_pages;
    A.L = make_layout(p); A.qnorm = qnorm; A.packed_lens = packed_lens;
    A.inv_pruned = p.keep < kHeadDim ? 1.0 / static_cast<double>(kHeadDim - p.keep) : 0.0;
    A.sel = make_select(p);
    A.status = static_cast<int*>(workspace);
    Bk.n_new = n_new;
    Bk.n_fresh = (n_new + kPageTokens - 1) / kPageTokens + 1;
    const int clear_warps = Bk.n_fresh < kBlockWarps ? Bk.n_fresh : kBlockWarps, warps = n_new < kBlockWarps ? n_new : kBlockWarps;
    launch_kernel(append_block_clear_kernel, dim3(p.n_kv_heads, p.batch, (Bk.n_fresh + clear_warps - 1) / clear_warps), dim3(32 * clear_warps), 0, stream, Bk);
    const dim3 grid(p.n_kv_heads, p.batch, (n_new + warps - 1) / warps), block(32 * warps);
    const bool rank = p.select != SPARK_SELECT_FIXED;
    if (p.dtype == SPARK_BF16) {
        if (rank) launch_kernel(append_block_token_kernel<__nv_bfloat16, true>, grid, block, 0, stream, Bk);
        else launch_kernel(append_block_token_kernel<__nv_bfloat16, false>, grid, block, 0, stream, Bk);
    } else {
        if (rank) launch_kernel(append_block_token_kernel<float, true>, grid, block, 0, stream, Bk);
        else launch_kernel(append_block_token_kernel<float, false>, grid, block, 0, stream, Bk);
    }
    launch_kernel(append_block_advance_kernel, dim3((p.batch + 127) / 128), dim3(128), 0, stream, Bk);
    *launches += 3;
    return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------
// Two partial attention results over disjoint token sets -> the result over their union (the log-sum-exp
// merge that split decoding uses, exposed for callers that hold a sequence in more than one cache).
// One warp per (sequence, query head) row; lane l owns channels 4l .. 4l+3.
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) merge_attn_kernel(int rows, const float* __restrict__ out_a, const float* __restrict__ lse_a,
                                                         const float* __restrict__ out_b, const float* __restrict__ lse_b,
                                                         float* __restrict__ out, float* __restrict__ lse)
{
    grid_wait();
    grid_release();
    const int row = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= rows) return;
    const float la = lse_a[row], lb = lse_b[row];
    const float m = fmaxf(la, lb);
    float wa = 0.f, wb = 0.f, l = -INFINITY;
    if (m > -INFINITY) {                                       // at least one side saw tokens
        const float ea = expf(la - m), eb = expf(lb - m);
        const float inv = 1.0f / (ea + eb);
        wa = ea * inv; wb = eb * inv;
        l = m + logf(ea + eb);
    }
    const float4 a = reinterpret_cast<const float4*>(out_a + static_cast<int64_t>(row) * kHeadDim)[lane];
    const float4 b = reinterpret_cast<const float4*>(out_b + static_cast<int64_t>(row) * kHeadDim)[lane];
    reinterpret_cast<float4*>(out + static_cast<int64_t>(row) * kHeadDim)[lane] =
        make_float4(fmaf(wa, a.x, wb * b.x), fmaf(wa, a.y, wb * b.y), fmaf(wa, a.z, wb * b.z), fmaf(wa, a.w, wb * b.w));
    if (lane == 0 && lse) lse[row] = l;
}

spark_status launch_merge_attn(int rows, const float* out_a, const float* lse_a, const float* out_b, const float* lse_b,
                               float* out, float* lse, cudaStream_t stream)
{
    if (rows == 0) return SPARK_OK;
    launch_kernel(merge_attn_kernel, dim3((rows + 3) / 4), dim3(128), 0, stream, rows, out_a, lse_a, out_b, lse_b, out, lse);
    return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------
// pages -> logical arrays
// ------------------------------------------------------------------------------------------------
template <int ES> struct ElemBits;
template <> struct ElemBits<2> { using type = unsigned short; };
template <> struct ElemBits<4> { using type = unsigned; };

struct UnpackArgs {
    const unsigned char* pages;
    const int32_t* block_table;
    int max_blocks;
    const int32_t* lens;
    int max_tokens;
    int Hkv;
    int64_t n_pool_pages;
    PageLayout L;
    uint32_t* mask;
    float* mu;
    void* vals;
    void* v;
    uint32_t* vmask;
    float* mu_all;
    float* sigma_all;
    int vec_vals, vec_v;          // rows of vals / v may be written 16 bytes at a time
};

// One CTA per page: the page comes into shared memory with 16-byte loads and every output array, whose 16 rows of a
// page are one contiguous piece, is written 16 bytes per thread (element by element only where its rows or its base are
// not 16-byte aligned).  What bounds it: the arrays it writes.  With divisions and 2-byte accesses per element the
// 8 heads x 12.4 K tokens of a batch of short prompts took 78 us, this 25 us (105 MB written, the pages partly from L2).
constexpr int kUnpackThreads = 128;

template <int ES>
__global__ void __launch_bounds__(kUnpackThreads) unpack_pages_kernel(UnpackArgs A)
{
    extern __shared__ __align__(16) unsigned char up_page[];
    using Elt = typename ElemBits<ES>::type;
    constexpr int kVec = 16 / ES;                              // elements per 16-byte store
    grid_wait();
    grid_release();
    const int blk = blockIdx.x, h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    const PageLayout L = A.L;
    const int T = L.keep;
    int len = A.lens[b];
    len = len < 0 ? 0 : (len > A.max_tokens ? A.max_tokens : len);
    const int64_t unit = static_cast<int64_t>(b) * A.Hkv + h;
    const int t0 = blk * kPageTokens;
    const int rows = min(kPageTokens, A.max_tokens - t0);      // rows of the outputs
    int live = len - t0;                                       // rows with a token
    live = live < 0 ? 0 : (live > rows ? rows : live);
    if (live > 0) {
        const int64_t id = A.block_table ? A.block_table[unit * A.max_blocks + blk] : unit * A.max_blocks + blk;
        if (id >= 0 && id < A.n_pool_pages) {
            const uint4* page = reinterpret_cast<const uint4*>(A.pages + id * L.page_bytes);
            for (int i = tid; i < L.page_bytes / 16; i += kUnpackThreads) reinterpret_cast<uint4*>(up_page)[i] = page[i];
        } else {
            live = 0;
        }
        __syncthreads();
    }
    const int64_t row0 = unit * A.max_tokens + t0;
    if (tid < rows * kMaskWords) {
        if (A.mask) A.mask[row0 * kMaskWords + tid] = tid < live * kMaskWords ? reinterpret_cast<const unsigned*>(up_page + L.mask_off)[tid] : 0u;
        if (A.vmask)                                           // all ones for dense value rows
            A.vmask[row0 * kMaskWords + tid] = tid >= live * kMaskWords ? 0u
                : (L.keep_v < kHeadDim ? reinterpret_cast<const unsigned*>(up_page + L.vmask_off)[tid] : 0xffffffffu);
    }
    if (tid < rows) {
        if (A.mu) A.mu[row0 + tid] = tid < live ? reinterpret_cast<const float*>(up_page + L.mu_off)[tid] : 0.f;
        const float* st = reinterpret_cast<const float*>(up_page + L.stats_off);      // only asked for where the section exists
        if (A.mu_all) A.mu_all[row0 + tid] = tid < live ? st[tid] : 0.f;
        if (A.sigma_all) A.sigma_all[row0 + tid] = tid < live ? st[kPageTokens + tid] : 0.f;
    }
    // thread (p, g): token p, element groups g, g + 8, ...
    const int p = tid & (kPageTokens - 1), g0 = tid >> 4;
    const bool on = p < live;
    if (A.vals && p < rows) {
        Elt* out = static_cast<Elt*>(A.vals) + (row0 + p) * T;
        const unsigned char* src = up_page + L.vals_off + val_offset(ES, p, 0);       // slot s is 16 elements further per step
        if (A.vec_vals) {
            for (int s0 = g0 * kVec; s0 < T; s0 += (kUnpackThreads / kPageTokens) * kVec) {
                alignas(16) Elt x[kVec];
#pragma unroll
                for (int e = 0; e < kVec; ++e)
                    x[e] = on ? *reinterpret_cast<const Elt*>(src + (s0 + e) * (kPageTokens * ES)) : static_cast<Elt>(0);
                *reinterpret_cast<uint4*>(out + s0) = *reinterpret_cast<const uint4*>(x);
            }
        } else {
            for (int s0 = g0; s0 < T; s0 += kUnpackThreads / kPageTokens)
                out[s0] = on ? *reinterpret_cast<const Elt*>(src + s0 * (kPageTokens * ES)) : static_cast<Elt>(0);
        }
    }
    if (A.v && L.keep_v >= kHeadDim) {                         // dense value rows: 16-byte chunks, lanes along a row
        for (int i = tid; i < rows * (kHeadDim / kVec); i += kUnpackThreads) {
            const int r = i / (kHeadDim / kVec), c = i % (kHeadDim / kVec);
            uint4 x = make_uint4(0, 0, 0, 0);
            if (r < live) x = *reinterpret_cast<const uint4*>(up_page + L.v_off + v_chunk_offset(ES, r, c));
            Elt* out = static_cast<Elt*>(A.v) + (row0 + r) * kHeadDim + c * kVec;
            if (A.vec_v) *reinterpret_cast<uint4*>(out) = x;
            else
                for (int e = 0; e < kVec; ++e) out[e] = reinterpret_cast<const Elt*>(&x)[e];
        }
    } else if (A.v && p < rows) {                              // kept value entries; pruned ones read back as zero
        const unsigned* vm = reinterpret_cast<const unsigned*>(up_page + L.vmask_off) + p * kMaskWords;
        Elt* row = static_cast<Elt*>(A.v) + (row0 + p) * kHeadDim;
        for (int c = g0; c < kHeadDim / kVec; c += kUnpackThreads / kPageTokens) {
            const int j0 = c * kVec;
            alignas(16) Elt x[kVec];
            unsigned word = on ? vm[j0 >> 5] : 0u;
            int slot = __popc(word & ((1u << (j0 & 31)) - 1u));
            if (on)
                for (int w = 0; w < (j0 >> 5); ++w) slot += __popc(vm[w]);
#pragma unroll
            for (int e = 0; e < kVec; ++e) {
                const bool kept = (word >> ((j0 + e) & 31)) & 1u;
                x[e] = kept ? *reinterpret_cast<const Elt*>(up_page + L.v_off + val_offset(ES, p, slot)) : static_cast<Elt>(0);
                slot += kept ? 1 : 0;
            }
            if (A.vec_v) *reinterpret_cast<uint4*>(row + j0) = *reinterpret_cast<const uint4*>(x);
            else
                for (int e = 0; e < kVec; ++e) row[j0 + e] = x[e];
        }
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
// Threads of the window norm per (sequence, KV head) with `rows` window rows.  Few units: as many as shorten the chain of
// loads (the page kernel of 1 x 32768 tokens waits for it: 65.7, 63.5, 61.3 us a prefill with 128, 256, 512).  Many units:
// as many as keep them resident together (us per prefill of one-token prompts with 128, 256, 512 threads: 512 units x 64
// rows 12.4, 12.4, 15.8; 1024 x 128 18.5, 19.4, 27.4; 512 x 512 34.7, 22.6, 22.7; 4096 x 16 39, 49, 74).  fp32 rows take
// twice the threads (512 x 64: 15.2, 14.8, 13.3; 1024 x 64: 16.7, 16.1, 17.8; 4096 x 16: 38, 43, 51).
inline int qnorm_threads(int64_t units, int rows, bool bf16)
{
    if (!bf16) return units <= 512 ? 512 : 128;
    return units <= 256 ? 512 : (rows > 128 ? 256 : 128);
}

// Released at its top, the window norm lets the page kernel become resident beside it and load keys and values meanwhile.
// With a CTA of the norm on half the SMs or more, a small page kernel's CTAs crowd onto the SMs that are left, so it is let in
// at the end (16 x 60 tokens with 8 KV heads: 18.7 us a prefill released at the top, 11.9 at the end; 16 x 200 18.8 and 17.3).
// A page kernel that fills every SM anyway, or a long norm, is better let in early (16 x 400: 20.9 and 21.8; 32 x 100 with
// 512 window rows: 23.0 and 25.3).
inline bool qnorm_release_early(int64_t units, int rows, int n_blocks)
{
    const int64_t page_ctas = units * ((n_blocks + kWarpPageWarps - 1) / kWarpPageWarps);
    return units <= 64 || rows > 256 || page_ctas > 740;
}

size_t compress_workspace_bytes(const spark_params& p, int64_t max_seq_tokens)
{
    return kWorkspaceHeader + evict_workspace_bytes(p, max_seq_tokens);
}

spark_status launch_compress(const spark_params& p, const void* q_win, const void* k, const void* v,
                             int64_t sb, int64_t sh, int64_t st, const int32_t* seq_lens,
                             int32_t max_seq_tokens, void* pages, const int32_t* block_table,
                             int32_t max_blocks, float* qnorm, int32_t* packed_lens, int32_t* kept_tokens,
                             void* workspace, size_t workspace_bytes, cudaStream_t stream, int* launches)
{
    (void)workspace_bytes;
    int* status = static_cast<int*>(workspace);
    const bool evict = p.token_budget > 0;
    const int64_t units = static_cast<int64_t>(p.batch) * p.n_kv_heads;
    if (evict) {            // writes kept_tokens, packed_lens and, where norm_in_select, qnorm
        const spark_status st_e = launch_evict(p, q_win, k, sb, sh, st, seq_lens, max_seq_tokens, qnorm, packed_lens,
                                               kept_tokens, workspace, stream, launches);
        if (st_e != SPARK_OK) return st_e;
    }
    const int max_packed = (evict && p.token_budget < max_seq_tokens) ? p.token_budget : max_seq_tokens;
    const int n_blocks = (max_packed + kPageTokens - 1) / kPageTokens;
    const float eps = norm_floor(p);
    const dim3 qgrid(p.n_kv_heads, p.batch);
    const int rows = p.n_q_heads / p.n_kv_heads * p.window;
    auto window_norm = [&](auto elem, auto threads, auto early) {
        constexpr int kThreads = decltype(threads)::value;
        launch_kernel(window_qnorm_kernel<decltype(elem), kThreads, decltype(early)::value>, qgrid, dim3(kThreads), 0, stream, q_win, p.n_q_heads,
                      p.n_kv_heads, p.window, eps, qnorm, seq_lens, evict ? nullptr : packed_lens, max_seq_tokens, status);
    };
    auto by_threads = [&](auto elem, auto early) {
        const int n = qnorm_threads(units, rows, p.dtype == SPARK_BF16);
        if (n == 128) window_norm(elem, std::integral_constant<int, 128>(), early);
        else if (n == 256) window_norm(elem, std::integral_constant<int, 256>(), early);
        else window_norm(elem, std::integral_constant<int, 512>(), early);
    };
    auto by_release = [&](auto elem) {
        if (qnorm_release_early(units, rows, n_blocks)) by_threads(elem, std::true_type());
        else by_threads(elem, std::false_type());
    };
    if (!evict || !norm_in_select(units)) {
        if (p.dtype == SPARK_BF16) by_release(__nv_bfloat16());
        else by_release(0.f);
        ++*launches;
        if (cudaGetLastError() != cudaSuccess) return SPARK_ERR_CUDA;
    }
    if (n_blocks == 0) return SPARK_OK;
    CompressArgs A;
    A.k = k; A.v = v; A.sb = sb; A.sh = sh; A.st = st;
    A.lens = packed_lens; A.gather = evict ? kept_tokens : nullptr; A.gather_stride = evict ? p.token_budget : 0;
    A.qnorm = qnorm; A.pages = static_cast<unsigned char*>(pages);
    A.block_table = block_table; A.max_blocks = max_blocks; A.Hkv = p.n_kv_heads; A.keep = p.keep;
    A.n_pool_pages = p.n_pool_pages; A.L = make_layout(p); A.status = status;
    A.inv_pruned = p.keep < kHeadDim ? 1.0 / static_cast<double>(kHeadDim - p.keep) : 0.0;
    A.sel = make_select(p);
    A.max_len = max_packed;
    const bool pv = A.L.keep_v < kHeadDim, topp = p.select == SPARK_SELECT_TOP_P;
    if (p.dtype == SPARK_BF16 && p.recovery == SPARK_RECOVER_DEGENERATE && (p.select == SPARK_SELECT_FIXED || (topp && !pv))) {
        if (!evict) A.lens = seq_lens;                         // readable before the window norm has ended
        const int per_cta = n_blocks == 1 ? 1 : (topp ? kToppWarps / 2 : kWarpPageWarps);         // pages
        const dim3 wgrid((n_blocks + per_cta - 1) / per_cta, p.n_kv_heads, p.batch);
        static unsigned char smem_raised[2][kMaxDevices] = {};                // (a single page needs less than the limit)
        cudaError_t e;
        if (topp) {                                            // (two pages: at most 19 KB)
            auto kernel = per_cta == 1 ? compress_topp_kernel<2> : compress_topp_kernel<kToppWarps>;
            e = launch_kernel(kernel, wgrid, dim3(per_cta * 64), 4 * kToppStride * 4 + per_cta * topp_page_room(A.L), stream, A);
        } else {
            const size_t smem = kHeadDim * 4 + per_cta * (kWarpPageFixed + static_cast<size_t>(pv ? A.L.page_bytes : A.L.v_off));
            auto pick = [&](auto w) {
                constexpr int kWarps = decltype(w)::value;
                return pv ? compress_pages_warp_kernel<true, kWarps> : compress_pages_warp_kernel<false, kWarps>;
            };
            auto kernel = per_cta == 1 ? pick(std::integral_constant<int, 1>()) : pick(std::integral_constant<int, kWarpPageWarps>());
            if (smem > 48 * 1024 && !allow_max_smem(kernel, smem_raised[pv ? 1 : 0])) return SPARK_ERR_CUDA;
            e = launch_kernel(kernel, wgrid, dim3(per_cta * 32), smem, stream, A);
        }
        ++*launches;
        return e == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
    }
    const dim3 grid(n_blocks, p.n_kv_heads, p.batch);
    const bool rank = p.select != SPARK_SELECT_FIXED;      // a ratio-free rule: the kernels with the rank sort
    if (p.dtype == SPARK_BF16) {
        if (rank) launch_kernel(compress_pages_kernel<__nv_bfloat16>, grid, dim3(256), A.L.page_bytes, stream, A);
        else launch_kernel(compress_pages4_kernel<__nv_bfloat16>, grid, dim3(128), A.L.page_bytes, stream, A);
    } else {
        if (rank) launch_kernel(compress_pages_kernel<float>, grid, dim3(256), A.L.page_bytes, stream, A);
        else launch_kernel(compress_pages4_kernel<float>, grid, dim3(128), A.L.page_bytes, stream, A);
    }
    ++*launches;
    if (cudaGetLastError() != cudaSuccess) return SPARK_ERR_CUDA;
    return SPARK_OK;
}

spark_status launch_unpack(const spark_params& p, const void* pages, const int32_t* block_table,
                           int32_t max_blocks, const int32_t* packed_lens, int32_t max_tokens,
                           uint32_t* mask, float* mu, void* vals, void* v, uint32_t* vmask, float* mu_all,
                           float* sigma_all, cudaStream_t stream)
{
    const int n_blocks = (max_tokens + kPageTokens - 1) / kPageTokens;
    if (n_blocks == 0) return SPARK_OK;
    UnpackArgs A;
    A.pages = static_cast<const unsigned char*>(pages); A.block_table = block_table;
    A.max_blocks = max_blocks; A.lens = packed_lens; A.max_tokens = max_tokens; A.Hkv = p.n_kv_heads;
    A.n_pool_pages = p.n_pool_pages; A.L = make_layout(p);
    A.mask = mask; A.mu = mu; A.vals = vals; A.v = v; A.vmask = vmask; A.mu_all = mu_all; A.sigma_all = sigma_all;
    A.vec_vals = (reinterpret_cast<uintptr_t>(vals) & 15) == 0 && (p.keep * A.L.esize & 15) == 0;
    A.vec_v = (reinterpret_cast<uintptr_t>(v) & 15) == 0;
    const dim3 grid(n_blocks, p.n_kv_heads, p.batch);           // (a page is at most 17 KB)
    if (A.L.esize == 2) launch_kernel(unpack_pages_kernel<2>, grid, dim3(kUnpackThreads), A.L.page_bytes, stream, A);
    else launch_kernel(unpack_pages_kernel<4>, grid, dim3(kUnpackThreads), A.L.page_bytes, stream, A);
    if (cudaGetLastError() != cudaSuccess) return SPARK_ERR_CUDA;
    return SPARK_OK;
}

}  // namespace spark
