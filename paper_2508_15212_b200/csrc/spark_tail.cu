// The dense tail of a sequence: recently appended tokens whose keys keep every channel (Sec. "Preliminaries",
// K <- Cat[K, k] taken literally).  Two kernels: one appends a token, one attends over a short tail; the merge with the
// pruned prefix happens in the prefix's decode step.
#include "spark_common.cuh"

namespace spark {

constexpr unsigned kTailMask = 0xffffffffu;

// ------------------------------------------------------------------------------------------------
// One new token per sequence into the tail's pages (keep = 128: every channel kept, mu = 0) and, as plain rows, into
// k_tail / v_tail [B][Hkv][cap][D]; the length advances.  A CTA per sequence, warps share its KV heads; every thread
// reads the length before the first barrier and thread 0 advances it after the second.
//   One launch of about 3 us; a page append that searched 128 of 128 channels and two strided copies took three (5 + 2 + 2).
// ------------------------------------------------------------------------------------------------
struct AppendDenseArgs {
    const void* k_new;
    const void* v_new;
    unsigned char* pages;
    const int32_t* block_table;
    int max_blocks, Hkv, cap;
    int64_t n_pool_pages;
    PageLayout L;
    void* k_tail;
    void* v_tail;
    int32_t* lens;
    int* status;
};

template <typename E>
__global__ void __launch_bounds__(1024) append_dense_kernel(AppendDenseArgs A)
{
    constexpr int kEs = sizeof(E), kLaneBytes = 4 * kEs;       // a lane owns channels 4*lane .. 4*lane+3
    using Vec = typename LaneVec<kEs>::type;
    grid_wait();
    grid_release();
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    const PageLayout L = A.L;
    // the first head's row before the length: one round trip less in the chain
    Vec k_first, v_first;
    if (warp < A.Hkv) {
        const int64_t first = (static_cast<int64_t>(b) * A.Hkv + warp) * 32 + lane;
        k_first = *reinterpret_cast<const Vec*>(static_cast<const unsigned char*>(A.k_new) + first * kLaneBytes);
        v_first = *reinterpret_cast<const Vec*>(static_cast<const unsigned char*>(A.v_new) + first * kLaneBytes);
    }
    const int t = A.lens[b];
    __syncthreads();
    const int blk = t / kPageTokens, p = t - blk * kPageTokens;
    const bool room = t >= 0 && t < A.cap && blk < A.max_blocks;
    if (!room && threadIdx.x == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
    for (int h = warp; room && h < A.Hkv; h += n_warps) {
        const int64_t unit = static_cast<int64_t>(b) * A.Hkv + h;
        const int64_t entry = unit * A.max_blocks + blk;
        const int64_t page_id = A.block_table ? A.block_table[entry] : entry;
        if (page_id < 0 || page_id >= A.n_pool_pages) {
            if (lane == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
            continue;
        }
        Vec k = k_first, v = v_first;
        if (h != warp) {
            k = *reinterpret_cast<const Vec*>(static_cast<const unsigned char*>(A.k_new) + (unit * 32 + lane) * kLaneBytes);
            v = *reinterpret_cast<const Vec*>(static_cast<const unsigned char*>(A.v_new) + (unit * 32 + lane) * kLaneBytes);
        }
        const int64_t row = unit * A.cap + t;
        *reinterpret_cast<Vec*>(static_cast<unsigned char*>(A.k_tail) + (row * 32 + lane) * kLaneBytes) = k;
        *reinterpret_cast<Vec*>(static_cast<unsigned char*>(A.v_tail) + (row * 32 + lane) * kLaneBytes) = v;
        unsigned char* page = A.pages + page_id * L.page_bytes;
        if (p == 0) {                                          // first token of a page: clear it
            for (int i = lane; i < L.page_bytes / 16; i += 32) reinterpret_cast<uint4*>(page)[i] = make_uint4(0, 0, 0, 0);
            __syncwarp();
        }
        const E* ke = reinterpret_cast<const E*>(&k);
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<E*>(page + L.vals_off + val_offset(kEs, p, 4 * lane + i)) = ke[i];
        const int c = lane * kLaneBytes / 16;                  // 16-byte chunk of the value row
        *reinterpret_cast<Vec*>(page + L.v_off + v_chunk_offset(kEs, p, c) + (lane * kLaneBytes & 15)) = v;
        if (lane < kMaskWords) reinterpret_cast<unsigned*>(page + L.mask_off)[p * kMaskWords + lane] = 0xffffffffu;
        if (lane == 0) reinterpret_cast<float*>(page + L.mu_off)[p] = 0.f;
    }
    __syncthreads();
    if (threadIdx.x == 0 && room) A.lens[b] = t + 1;
}

// ------------------------------------------------------------------------------------------------
// Attention over a tail of at most kTailMax tokens, a CTA per (sequence, KV head): four threads per token for the scores
// (32 channels each, all G heads from one read of the key), a warp per head for the softmax, then four token groups by 64
// channel pairs for the weighted sum.  fp32 storage sums its scores in double, as the page kernel does.
//   Latency bound (a few dependent rounds over 16 KB): about 4 us where the page kernel, whose start and merge are laid out
//   for long caches, took 8 us for the same 64 tokens; longer tails stay with that kernel.
// ------------------------------------------------------------------------------------------------
constexpr int kTailThreads = 256;

template <int ES> struct TailPair;
template <> struct TailPair<2> { using type = unsigned; };
template <> struct TailPair<4> { using type = uint2; };

struct TailArgs {
    const void* q;
    const void* k;
    const void* v;
    const int32_t* lens;
    int Hq, Hkv, cap;
    float scale_log2e;
    float* out;
    float* lse;
    int* status;
};

template <int G, typename E>
__global__ void __launch_bounds__(kTailThreads) tail_attn_kernel(TailArgs A)
{
    using Acc = typename TailAcc<E>::type;
    __shared__ __align__(16) float q_s[G][kHeadDim];
    __shared__ float prob[G][kTailMax];
    __shared__ float norm[G];
    __shared__ __align__(16) float part[4][G][kHeadDim];
    grid_wait();
    grid_release();
    const int h = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // rows of the first 64 tokens before the length is known (they exist up to cap; what is past the length is not used)
    const int64_t unit = static_cast<int64_t>(b) * A.Hkv + h, row0 = static_cast<int64_t>(b) * A.Hq + h * G;
    const E* k = static_cast<const E*>(A.k) + unit * A.cap * kHeadDim;
    const E* v = static_cast<const E*>(A.v) + unit * A.cap * kHeadDim;
    constexpr int kVecs = 32 * sizeof(E) / 16;
    using Pair = typename TailPair<sizeof(E)>::type;
    const int t0 = tid >> 2, c = tid & 3, grp = tid >> 6, c2 = tid & 63;
    uint4 kr[kVecs];
    Pair vr[16];
    if (t0 < A.cap)
#pragma unroll
        for (int i = 0; i < kVecs; ++i) kr[i] = reinterpret_cast<const uint4*>(k + static_cast<int64_t>(t0) * kHeadDim + 32 * c)[i];
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (grp + 4 * i < A.cap) vr[i] = *reinterpret_cast<const Pair*>(v + static_cast<int64_t>(grp + 4 * i) * kHeadDim + 2 * c2);
    int n = A.lens[b];
    if (n < 0 || n > A.cap) {
        if (tid == 0 && h == 0) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
        n = n < 0 ? 0 : A.cap;
    }
    for (int i = tid; i < G * kHeadDim; i += kTailThreads) q_s[i / kHeadDim][i % kHeadDim] = Elem<E>::load(A.q, row0 * kHeadDim + i);
    __syncthreads();
    for (int t = t0; t < ((n + 63) & ~63); t += 64) {          // whole warps iterate together
        const bool on = t < n;
        if (t >= 64 && on)
#pragma unroll
            for (int i = 0; i < kVecs; ++i) kr[i] = reinterpret_cast<const uint4*>(k + static_cast<int64_t>(t) * kHeadDim + 32 * c)[i];
        Acc s[G];
#pragma unroll
        for (int g = 0; g < G; ++g) s[g] = 0;
        if (on)
#pragma unroll
            for (int i = 0; i < kVecs; ++i) {
                constexpr int kPer = 16 / sizeof(E);
                const E* x = reinterpret_cast<const E*>(&kr[i]);
                float f[kPer];
#pragma unroll
                for (int e = 0; e < kPer; ++e) f[e] = static_cast<float>(x[e]);
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int e = 0; e < kPer; e += 4) {
                        const float4 qq = *reinterpret_cast<const float4*>(&q_s[g][32 * c + i * kPer + e]);
                        s[g] += static_cast<Acc>(f[e]) * static_cast<Acc>(qq.x);
                        s[g] += static_cast<Acc>(f[e + 1]) * static_cast<Acc>(qq.y);
                        s[g] += static_cast<Acc>(f[e + 2]) * static_cast<Acc>(qq.z);
                        s[g] += static_cast<Acc>(f[e + 3]) * static_cast<Acc>(qq.w);
                    }
            }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            s[g] += __shfl_xor_sync(kTailMask, s[g], 1);
            s[g] += __shfl_xor_sync(kTailMask, s[g], 2);
            if (c == 0) prob[g][t] = on ? static_cast<float>(s[g] * static_cast<Acc>(A.scale_log2e)) : -INFINITY;
        }
    }
    __syncthreads();
    if (warp < G) {
        float x[kTailMax / 32], m = -INFINITY, l = 0.f;
#pragma unroll
        for (int i = 0; i < kTailMax / 32; ++i) {
            x[i] = lane + 32 * i < n ? prob[warp][lane + 32 * i] : -INFINITY;
            m = fmaxf(m, x[i]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kTailMask, m, o));
#pragma unroll
        for (int i = 0; i < kTailMax / 32; ++i) {
            const float e = x[i] == -INFINITY ? 0.f : exp2f(x[i] - m);
            if (lane + 32 * i < n) prob[warp][lane + 32 * i] = e;
            l += e;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(kTailMask, l, o);
        if (lane == 0) {
            norm[warp] = n > 0 ? 1.0f / l : 0.f;
            A.lse[row0 + warp] = n > 0 ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
        }
    }
    __syncthreads();
    // weighted sum: tokens grp, grp + 4, ...; channels 2*c2, 2*c2 + 1
    float2 acc[G];
#pragma unroll
    for (int g = 0; g < G; ++g) acc[g] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int t = grp + 4 * i;
        if (t >= n) break;
        const E* x = reinterpret_cast<const E*>(&vr[i]);
        const float v0 = static_cast<float>(x[0]), v1 = static_cast<float>(x[1]);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            acc[g].x = fmaf(prob[g][t], v0, acc[g].x);
            acc[g].y = fmaf(prob[g][t], v1, acc[g].y);
        }
    }
#pragma unroll 8
    for (int t = 64 + grp; t < n; t += 4) {
        const E* x = v + static_cast<int64_t>(t) * kHeadDim + 2 * c2;
        const float v0 = static_cast<float>(x[0]), v1 = static_cast<float>(x[1]);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            acc[g].x = fmaf(prob[g][t], v0, acc[g].x);
            acc[g].y = fmaf(prob[g][t], v1, acc[g].y);
        }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) *reinterpret_cast<float2*>(&part[grp][g][2 * c2]) = acc[g];
    __syncthreads();
    for (int i = tid; i < G * kHeadDim; i += kTailThreads) {
        const int g = i / kHeadDim, j = i % kHeadDim;
        A.out[row0 * kHeadDim + i] = ((part[0][g][j] + part[1][g][j]) + (part[2][g][j] + part[3][g][j])) * norm[g];
    }
}

spark_status launch_append_dense(const spark_params& p, const void* k_new, const void* v_new, void* pages,
                                 const int32_t* block_table, int32_t max_blocks, void* k_tail, void* v_tail, int32_t cap,
                                 int32_t* packed_lens, void* workspace, cudaStream_t stream, int* launches)
{
    AppendDenseArgs A;
    A.k_new = k_new; A.v_new = v_new; A.pages = static_cast<unsigned char*>(pages); A.block_table = block_table;
    A.max_blocks = max_blocks; A.Hkv = p.n_kv_heads; A.cap = cap; A.n_pool_pages = p.n_pool_pages;
    A.L = make_layout(p); A.k_tail = k_tail; A.v_tail = v_tail; A.lens = packed_lens;
    A.status = static_cast<int*>(workspace);
    const dim3 block(32 * (p.n_kv_heads < 32 ? p.n_kv_heads : 32));
    const cudaError_t e = p.dtype == SPARK_BF16 ? launch_kernel(append_dense_kernel<__nv_bfloat16>, dim3(p.batch), block, 0, stream, A)
                                                : launch_kernel(append_dense_kernel<float>, dim3(p.batch), block, 0, stream, A);
    ++*launches;
    return e == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

template <int G> static cudaError_t launch_tail_g(const spark_params& p, const TailArgs& A, cudaStream_t stream)
{
    const dim3 grid(p.n_kv_heads, p.batch);
    return p.dtype == SPARK_BF16 ? launch_kernel(tail_attn_kernel<G, __nv_bfloat16>, grid, dim3(kTailThreads), 0, stream, A)
                                 : launch_kernel(tail_attn_kernel<G, float>, grid, dim3(kTailThreads), 0, stream, A);
}

spark_status launch_tail_attn(const spark_params& p, const void* q, const void* k_tail, const void* v_tail, int32_t cap,
                              const int32_t* tail_lens, float* out, float* lse, void* workspace, cudaStream_t stream, int* launches)
{
    TailArgs A;
    A.q = q; A.k = k_tail; A.v = v_tail; A.lens = tail_lens; A.Hq = p.n_q_heads; A.Hkv = p.n_kv_heads; A.cap = cap;
    const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 1.0f / sqrtf(static_cast<float>(p.head_dim));
    A.scale_log2e = scale * 1.4426950408889634f;
    A.out = out; A.lse = lse; A.status = static_cast<int*>(workspace);
    cudaError_t e = cudaErrorInvalidValue;
    switch (p.n_q_heads / p.n_kv_heads) {
        case 1: e = launch_tail_g<1>(p, A, stream); break;
        case 2: e = launch_tail_g<2>(p, A, stream); break;
        case 3: e = launch_tail_g<3>(p, A, stream); break;
        case 4: e = launch_tail_g<4>(p, A, stream); break;
        case 5: e = launch_tail_g<5>(p, A, stream); break;
        case 6: e = launch_tail_g<6>(p, A, stream); break;
        case 7: e = launch_tail_g<7>(p, A, stream); break;
        case 8: e = launch_tail_g<8>(p, A, stream); break;
    }
    ++*launches;
    return e == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace spark
