// Shared declarations of the SparK CUDA library: page layout, status word, small device helpers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/spark.h"

namespace spark {

constexpr int kHeadDim = 128;        // D
constexpr int kPageTokens = 16;      // P
constexpr int kMaskWords = 4;        // 128-bit channel mask per token
constexpr int kMaxGroup = 8;         // G = Hq / Hkv
constexpr int kMaxBatch = 1024;      // sequences per call (decode keeps a per-sequence prefix in shared memory)
constexpr int kMaxCtas = 256;        // upper bound of the persistent decode grid (sizes the partial-result slots)
constexpr int kWorkspaceHeader = 256;

// Byte layout of one page (16 tokens of one KV head).  Private to the library.
//
//   vals : T rows of 16 elements.  Row s holds kept slot s of every token; slot s of a token is its
//          s-th kept channel in ascending channel order.  Rows are 32 bytes (bf16) or 64 bytes (fp32), so
//          the section is exactly T elements per token.  In fp32 rows token p sits at element p; in bf16
//          rows at element (p & 7) * 2 + (p >> 3), so the eight tokens that one half of a matrix
//          fragment reads together fall into eight different 4-byte banks.
//   mask : [16][4] uint32, bit (j % 32) of word (j / 32) set <=> channel j kept
//   mu   : [16] float, mean saliency of the pruned channels
//   stats: (sampled recovery only) [16] float mean and [16] float population deviation of ALL the token's saliencies
//   v    : dense values (keep_v == 128): [16][128] elements, the value rows.  In bf16 pages the 16-byte
//          chunks of row p are stored at chunk index (c ^ (p & 7)), which makes the transposing matrix
//          loads of the decode kernel free of bank conflicts; fp32 pages store rows plainly.
//          pruned values (keep_v < 128): T_v rows of 16 elements laid out exactly like `vals` (slot s of
//          a token = its s-th kept value channel), followed by
//   vmask: [16][4] uint32 (pruned values only), bit (j % 32) of word (j / 32) set <=> value channel j kept
struct PageLayout {
    int vals_off;    // start of the kept key values (0, or behind everything else when `ragged`)
    int ragged;      // SparK-p pages: the slot rows come last and a per-page row count says how many are in use
    int esize;       // bytes per element (2 bf16, 4 fp32)
    int keep;        // T
    int keep_v;      // T_v (128: dense value rows)
    int mask_off;
    int mu_off;
    int stats_off;   // [16] float all-channel mean, [16] float population deviation (sampled recovery only)
    int recovery;    // spark_recovery
    int v_off;
    int vmask_off;   // meaningful when keep_v < 128
    int page_bytes;
};

// spark_params.keep_v -> T_v (0 and 128 both mean dense value rows)
__host__ __device__ inline int value_keep(int keep_v) { return (keep_v <= 0 || keep_v >= kHeadDim) ? kHeadDim : keep_v; }

// With SparK-p the number of kept channels varies per token, so a page's slot rows are only used up to the
// largest count among its 16 tokens.  Such pages are laid out with the slot rows LAST, and a row count per
// pool page (int32, in a side array behind the pages of the pool) tells the decode step how many bytes of the
// page to copy: mask | mu | (stats) | values | the first `rows` slot rows.
__host__ __device__ inline PageLayout make_layout(int dtype, int keep, int keep_v, int recovery, int ragged = 0)
{
    PageLayout L;
    L.esize = (dtype == SPARK_BF16) ? 2 : 4;
    L.keep = keep;
    L.keep_v = value_keep(keep_v);
    L.ragged = ragged;
    L.vals_off = 0;
    L.mask_off = ragged ? 0 : keep * kPageTokens * L.esize;
    L.mu_off = L.mask_off + kPageTokens * 16;
    L.stats_off = L.mu_off + kPageTokens * 4;
    L.recovery = recovery;
    L.v_off = L.stats_off + (recovery != SPARK_RECOVER_DEGENERATE ? 2 * kPageTokens * 4 : 0);
    L.vmask_off = L.v_off + L.keep_v * kPageTokens * L.esize;
    L.page_bytes = L.vmask_off + (L.keep_v < kHeadDim ? kPageTokens * 16 : 0);
    if (ragged) {
        L.vals_off = L.page_bytes;
        L.page_bytes += keep * kPageTokens * L.esize;
    }
    return L;
}

// the per-page row counts of a ragged pool: an int32 per pool page behind the pages (256-byte aligned)
__host__ __device__ inline int64_t rows_offset(int64_t n_pool_pages, int page_bytes)
{
    return (n_pool_pages * page_bytes + 255) / 256 * 256;
}

// byte offset of kept slot s of token p inside the vals section
__host__ __device__ inline int val_offset(int esize, int p, int s)
{
    return esize == 2 ? (s * kPageTokens + ((p & 7) * 2 + (p >> 3))) * 2 : (s * kPageTokens + p) * 4;
}

// byte offset (inside the v section) of the 16-byte chunk c of token p's value row
__host__ __device__ inline int v_chunk_offset(int esize, int p, int c)
{
    return esize == 2 ? (p * (kHeadDim * 2) + ((c ^ (p & 7)) << 4)) : (p * (kHeadDim * 4) + (c << 4));
}

// Workspace header: word 0 is the status word (first error wins).
__device__ inline void record_error(int* status, int code)
{
    atomicCAS(status, 0, code);
}

__device__ __forceinline__ float bf16_bits_to_float(unsigned short h)
{
    return __uint_as_float(static_cast<unsigned>(h) << 16);
}

template <typename E> struct Elem;
template <> struct Elem<float> {
    static constexpr int dtype = SPARK_F32;
    __device__ static float load(const void* p, int64_t i) { return static_cast<const float*>(p)[i]; }
};
template <> struct Elem<__nv_bfloat16> {
    static constexpr int dtype = SPARK_BF16;
    __device__ static float load(const void* p, int64_t i)
    {
        return bf16_bits_to_float(static_cast<const unsigned short*>(p)[i]);
    }
};

// four channels of a lane, and the type that sums the scores of a dense tail
template <int ES> struct LaneVec;
template <> struct LaneVec<2> { using type = uint2; };
template <> struct LaneVec<4> { using type = uint4; };
template <typename E> struct TailAcc;
template <> struct TailAcc<float> { using type = double; };
template <> struct TailAcc<__nv_bfloat16> { using type = float; };
constexpr int kTailMax = 128;         // tokens of a dense tail that tail_attn_kernel takes

// Programmatic dependent launch.  Every kernel of the library is launched so that it may become resident while the
// kernel before it on the stream drains (grid_release lets the next kernel become resident; grid_wait returns once the
// kernel before has completed and its writes are visible, at once under an ordinary predecessor), so that the launch
// latency and a kernel's own set-up run under the predecessor's last CTAs: back-to-back decode steps on one stream went
// from 27.0 to 25.4 us (1 x 32K tokens), from 14.35 to 12.7 us (fp32, 1024 tokens); append + decode 44.5 to 40.9 us.
//   Rule: a kernel releases only behind its own wait.  So a kernel that has started may rely on everything enqueued
// before its predecessor, and the order of a stream is unchanged for every kernel that waits at its top, before it
// touches anything of a caller's.  All do, with these exceptions, each of which reads early only what its predecessor
// cannot write:
//   - compress_pages_warp_kernel and compress_topp_kernel without eviction: keys, values, lengths and block table; behind the window norm;
//   - evict_scores_tc_kernel<2>: queries, keys and lengths; behind pass 1 of the same call;
//   - evict_select_kernel behind the second vote pass: window queries, and it writes the window norm, which that pass does not read;
//   - a decode step with SPARK_FLAG_OVERLAP_PREVIOUS: lengths, block table and pages; the caller vouches for the
//     predecessor.  Its consumers wait and release, not its producer (consumer_wait_previous);
//   - a decode step merged with a dense tail (late_wait): everything but the tail's result; behind tail_attn_kernel, which
//     writes nothing else.  The one kernel that releases before it waits: its successor may rely on everything enqueued
//     before the tail kernel, and not on the tail's result, which only this step reads.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// a[b][h][j] = max(|mean over the G*W window queries of the group|, eps) by the first kThreads threads of a CTA (the others
// only meet the barriers; `between` runs between the two): a thread sums 16 bytes' worth of channels over every 32nd (fp32: 16th)
// row of 512 threads in double, the row groups are then added in a fixed order.  (The sum is exact in double for any order unless its
// terms differ by more than 2^21.)  `part`: half as many rows of sums as there are row groups.
template <typename E, int kThreads, typename F>
__device__ __forceinline__ void window_norm(const void* __restrict__ q_win, int Hq, int Hkv, int W, float eps, float* __restrict__ qnorm,
                                            int h, int b, int tid, double (*part)[kHeadDim], F between)
{
    constexpr int kVec = 16 / sizeof(E);                       // channels per 16-byte load
    constexpr int kChunks = kHeadDim / kVec, kGroups = kThreads / kChunks;
    const int G = Hq / Hkv, rows = G * W;
    const int c = tid % kChunks, grp = tid / kChunks;
    const bool on = tid < kThreads;
    // the group's G*W window rows are consecutive in memory, (g outer, w inner)
    const E* src = static_cast<const E*>(q_win) + (static_cast<int64_t>(b) * Hq + h * G) * W * kHeadDim + c * kVec;
    double acc[kVec];
#pragma unroll
    for (int i = 0; i < kVec; ++i) acc[i] = 0.0;
    const bool aligned = (reinterpret_cast<uintptr_t>(q_win) & 15) == 0;
#pragma unroll 4
    for (int r = on ? grp : rows; r < rows; r += kGroups) {
        alignas(16) E x[kVec];
        const E* row = src + static_cast<int64_t>(r) * kHeadDim;
        if (aligned) *reinterpret_cast<uint4*>(x) = *reinterpret_cast<const uint4*>(row);
        else
            for (int i = 0; i < kVec; ++i) x[i] = row[i];
#pragma unroll
        for (int i = 0; i < kVec; ++i) acc[i] += static_cast<double>(static_cast<float>(x[i]));
    }
    if (on && grp >= kGroups / 2)
#pragma unroll
        for (int i = 0; i < kVec; ++i) part[grp - kGroups / 2][c * kVec + i] = acc[i];
    __syncthreads();
    if (grp < kGroups / 2)
#pragma unroll
        for (int i = 0; i < kVec; ++i) part[grp][c * kVec + i] += acc[i];
    between();
    __syncthreads();
    if (tid < kHeadDim) {
        double sum = 0.0;
#pragma unroll
        for (int g = 0; g < kGroups / 2; ++g) sum += part[g][tid];
        const float m = static_cast<float>(sum / static_cast<double>(rows));
        qnorm[(static_cast<int64_t>(b) * Hkv + h) * kHeadDim + tid] = fmaxf(fabsf(m), eps);
    }
}
// With eviction the window norm is done by the select kernel, under the vote pass's last CTAs, where all its CTAs (1024 threads each, two
// to an SM) are resident at once; with more units only the first of several rounds would hide it, and a launch of its own is
// better.  us per evicting prefill with a launch / in the select kernel: 1 x 131072 with 8 KV heads 154.2 / 153.3, 1 x 100000 with 4
// 122.6 / 119.1, 4 x 4000 64.1 / 61.5, 32 x 3000 (256 units) 199.8 / 198.0; 64 x 1000 (512) 166.7 / 175.6, 64 x 1500 294.6 / 300.3,
// 128 x 1500 (1024) 416 / 424.
inline bool norm_in_select(int64_t units) { return units <= 256; }
inline float norm_floor(const spark_params& p) { return p.qnorm_eps > 0.f ? p.qnorm_eps : 1e-12f; }

// Launch as a programmatic dependent, in clusters of `cluster` CTAs along x.
template <typename... Params, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(Params...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const Args&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <typename... Params, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const Args&... args)
{
    return launch_cluster(kernel, 1, grid, block, smem, stream, args...);
}

// Device properties the launchers need, looked up once per device and then served from a table
// (spark_decode.cu); `dev` is the current device.
constexpr int kMaxDevices = 64;
struct DeviceInfo { int n_sms; int smem_optin; };
bool device_info(int* dev, DeviceInfo* info);

// Raises a kernel's dynamic shared-memory limit to all that the device gives beside its static part, once per device and
// kernel.  (Setting it to what a launch needs, launch by launch, lets one thread lower it between another's call and launch.)
template <typename Kernel> inline bool allow_max_smem(Kernel kernel, int dev, int smem_optin, unsigned char (&done)[kMaxDevices])
{
    if (dev < 0 || dev >= kMaxDevices) return false;
    if (done[dev]) return true;                           // a racing first call only repeats the same setting
    cudaFuncAttributes at;
    if (cudaFuncGetAttributes(&at, kernel) != cudaSuccess) return false;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin - static_cast<int>(at.sharedSizeBytes)) != cudaSuccess)
        return false;
    done[dev] = 1;
    return true;
}
template <typename Kernel> inline bool allow_max_smem(Kernel kernel, unsigned char (&done)[kMaxDevices])
{
    int dev = 0;
    DeviceInfo info;
    return device_info(&dev, &info) && allow_max_smem(kernel, dev, info.smem_optin, done);
}

// host-side validation of a parameter block (spark_api.cu)
spark_status check_params(const spark_params* p);

// ---- host-side launchers implemented in the .cu files -------------------------------------------
spark_status launch_compress(const spark_params& p, const void* q_win, const void* k, const void* v,
                             int64_t sb, int64_t sh, int64_t st, const int32_t* seq_lens,
                             int32_t max_seq_tokens, void* pages, const int32_t* block_table,
                             int32_t max_blocks, float* qnorm, int32_t* packed_lens, int32_t* kept_tokens,
                             void* workspace, size_t workspace_bytes, cudaStream_t stream, int* launches);

spark_status launch_unpack(const spark_params& p, const void* pages, const int32_t* block_table,
                           int32_t max_blocks, const int32_t* packed_lens, int32_t max_tokens,
                           uint32_t* mask, float* mu, void* vals, void* v, uint32_t* vmask, float* mu_all,
                           float* sigma_all, cudaStream_t stream);
inline PageLayout make_layout(const spark_params& p)
{
    return make_layout(p.dtype, p.keep, p.keep_v, p.recovery, p.select == SPARK_SELECT_TOP_P ? 1 : 0);
}
int group_keep(int head_dim, int n_groups, const float* prune);

spark_status launch_decode(const spark_params& p, const void* q, const void* pages,
                           const int32_t* block_table, int32_t max_blocks, const int32_t* packed_lens,
                           const float* qnorm, float* out, float* lse, void* workspace,
                           size_t workspace_bytes, cudaStream_t stream, int* launches, bool q_by_value = false,
                           const float* other_out = nullptr, const float* other_lse = nullptr);
// other_out / other_lse: attention over further tokens of the same sequences, merged into the result.  The kernel that writes
// them must be the one enqueued just before, and must write nothing else that this step uses (the status word, which both
// only set by compare-and-swap, excepted): it is waited for only there.
// q_by_value: q is a HOST pointer and its bytes travel as a launch parameter (bf16 storage, degenerate recovery,
// dense value rows, at most query_by_value_limit() bytes; anything else is refused)
size_t query_by_value_limit();

spark_status launch_append(const spark_params& p, const void* k_new, const void* v_new, void* pages,
                           const int32_t* block_table, int32_t max_blocks, const float* qnorm,
                           int32_t* packed_lens, void* workspace, cudaStream_t stream, int* launches);

spark_status launch_append_block(const spark_params& p, const void* k_new, const void* v_new, int32_t n_new,
                                 void* pages, const int32_t* block_table, int32_t max_blocks, const float* qnorm,
                                 int32_t* packed_lens, void* workspace, cudaStream_t stream, int* launches);
spark_status launch_append_dense(const spark_params& p, const void* k_new, const void* v_new, void* pages,
                                 const int32_t* block_table, int32_t max_blocks, void* k_tail, void* v_tail, int32_t cap,
                                 int32_t* packed_lens, void* workspace, cudaStream_t stream, int* launches);
spark_status launch_tail_attn(const spark_params& p, const void* q, const void* k_tail, const void* v_tail, int32_t cap,
                              const int32_t* tail_lens, float* out, float* lse, void* workspace, cudaStream_t stream, int* launches);
spark_status launch_merge_attn(int rows, const float* out_a, const float* lse_a, const float* out_b, const float* lse_b,
                               float* out, float* lse, cudaStream_t stream);

size_t decode_workspace_bytes(const spark_params& p);
size_t evict_workspace_bytes(const spark_params& p, int64_t max_seq_tokens);
spark_status launch_evict(const spark_params& p, const void* q_win, const void* k, int64_t sb, int64_t sh,
                          int64_t st, const int32_t* seq_lens, int32_t max_seq_tokens, float* qnorm, int32_t* packed_lens,
                          int32_t* kept_tokens, void* workspace, cudaStream_t stream, int* launches);
size_t compress_workspace_bytes(const spark_params& p, int64_t max_seq_tokens);

}  // namespace spark
