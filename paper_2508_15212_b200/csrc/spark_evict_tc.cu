// Eviction votes on the 5th-generation tensor cores (tcgen05 + tensor memory), bf16 storage.
//
// The window-attention scores of the eviction pre-step are the one dense contraction of the method:
// per KV head, [G*W window-query rows x 128 channels] by [128 channels x S keys].  This file computes
// the same two passes as the CUDA-core kernels of spark_evict.cu with tcgen05.mma:
//   pass 1   D[row][token]  = Q . K^T   (M = 128 query rows, N = 128 keys per tile): a thread owns a
//            query row of the accumulator in tensor memory and keeps the row's running softmax max and
//            sum over all the tiles of its CTA -- no cross-thread reduction;
//   pass 2   D[token][row]  = K . Q^T   (M = 128 keys, N = padded row count <= 256): a thread owns a key
//            and adds up its probabilities over the query rows in a fixed order -- the votes are
//            reproducible and need no atomics.
// One warp feeds the tensor cores: key tiles come in by TMA (128-byte swizzle, the layout that the matrix descriptors name:
// row r of a 64-channel block at r*128 bytes, its 16-byte chunks XOR-ed with r & 7; 8-row groups 1024 bytes apart), tile i is
// multiplied into accumulator i & 1 as soon as its keys have landed and the accumulator has been read.  Two warpgroups per
// block of 128 query rows take the accumulators in turn, each a whole tile, so no barrier of the CTA stands in the loop: all
// hand-overs are mbarriers (the MMAs' through tcgen05.commit).  Every wait is bounded.
// What bounds it: the exponentials (1024 cycles of the SM's special function units per 128 x 128 scores, 68 % busy in pass 1, 58 % in
// pass 2), the keys' bytes (61 and 53 % of the DRAM's rate), then a CTA's start.  The passes over 8 x 131072 keys take 55 + 63 us one at a
// time from a cold cache, 67 + 65 with copies by all threads and a CTA barrier per tile.  Evicting prefill then -> now (the window norm in
// the select kernel too), builds in turn: 1 x 131072 174 -> 152 us, 1 x 100000 with 28 / 4 heads 154 -> 118, 2 x 30000 111 -> 98, 4 x 4000
// 71 -> 61.  A quarter of the exponentials as a polynomial on the FMA pipe was no faster, but for 2 us at 131072: not kept.
#include <cuda.h>

#include <type_traits>

#include "spark_common.cuh"

namespace spark {

constexpr int kTcTile = 128;            // keys per tile
constexpr unsigned long long kTcWaitNs = 1000000000ull;   // every device-side wait gives up after one second
// Blocks of 128 query rows: one or two.  Two warpgroups per block take turns in reading accumulators, one warp feeds the tensor cores.
__host__ __device__ constexpr int tc_threads(int blocks) { return blocks * 256 + 32; }
__host__ __device__ constexpr int tc_bufs(int blocks) { return blocks == 1 ? 2 : 4; }        // key buffers: two CTAs per SM with one row block, one with two

struct EvictTcArgs {
    const void* q_win;
    const void* k;
    int64_t sb, sh, st;
    const int32_t* seq_lens;
    int Hq, Hkv, W, budget;
    int S_max, tiles_per_cta, parts;     // parts = CTAs per unit
    int head_step, seq_step;             // tensor-map coordinates of the next head and sequence (0: the keys are shared)
    float* partial;      // [units][parts][R][2]   (pass 1 out, pass 2 in)
    float* votes;        // [units][S_max]
    int* status;
};

__device__ __forceinline__ unsigned tc_smem_u32(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }

// K-major, 128-byte swizzle: start address, stride between 8-row groups = 1024 bytes, descriptor version 1.
__device__ __forceinline__ uint64_t tc_desc(unsigned smem_addr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);            // bits [0,14)  start address >> 4
    d |= static_cast<uint64_t>(1) << 16;                                 // bits [16,30) leading byte offset (unused for swizzled K-major)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;                         // bits [32,46) stride byte offset >> 4
    d |= static_cast<uint64_t>(1) << 46;                                 // bits [46,48) descriptor version
    d |= static_cast<uint64_t>(2) << 61;                                 // bits [61,64) layout: 128-byte swizzle
    return d;
}

// kind::f16 instruction descriptor: D = f32, A = B = bf16, both K-major, shape M x N x 16.
__host__ __device__ constexpr unsigned tc_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<unsigned>(N >> 3) << 17) | (static_cast<unsigned>(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(unsigned d_tmem, uint64_t a_desc, uint64_t b_desc, unsigned idesc, unsigned accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ float tc_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 32 / 64 consecutive columns of this thread's tensor-memory lane: load and wait in a single statement, so nothing reads
// the registers before the wait.
__device__ __forceinline__ void tc_ld32(unsigned taddr, float (&v)[32])
{
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tc_ld64(unsigned taddr, float (&v)[64])
{
    unsigned r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]),
          "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]),
          "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]),
          "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]),
          "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}

// Copy `rows` rows of 128 bf16 channels (row i at src + i*stride elements; rows >= valid are zero) into
// the two 64-channel swizzled blocks at dst (block 0 at dst, block 1 at dst + rows_alloc*128 bytes).
__device__ __forceinline__ void tc_stage_rows(unsigned char* dst, int rows_alloc, const unsigned short* src, int64_t stride,
                                              int valid, int tid, int threads)
{
    for (int i = tid; i < rows_alloc * 16; i += threads) {
        const int r = i >> 4, ch16 = i & 15;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < valid) v = *reinterpret_cast<const uint4*>(src + static_cast<int64_t>(r) * stride + ch16 * 8);
        const int kb = ch16 >> 3, c8 = ch16 & 7;
        *reinterpret_cast<uint4*>(dst + static_cast<size_t>(kb) * rows_alloc * 128 + r * 128 + ((c8 ^ (r & 7)) << 4)) = v;
    }
}

// One 64-channel block of 128 key rows, swizzled as above, from the keys' tensor map (channel, token, head, sequence).
__device__ __forceinline__ void tc_load_keys(unsigned dst, const CUtensorMap* map, int channel, int token, int head, int seq, unsigned bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(map), "r"(channel), "r"(token), "r"(head), "r"(seq), "r"(bar)
        : "memory");
}

// Wait with a limit; on expiry (or when another thread gave up) the CTA's abort flag is set and the caller leaves its loop.
__device__ __forceinline__ bool tc_wait(unsigned bar, unsigned parity, volatile int* abort_flag)
{
    unsigned long long start = 0;
    for (unsigned it = 1;; ++it) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if (*abort_flag) return false;
        if ((it & 255u) == 0) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (start == 0) start = now;
            else if (now - start > kTcWaitNs) break;
        }
    }
    *abort_flag = 1;
    return false;
}

// pairs of fp32 in one instruction, and a maximum of three
__device__ __forceinline__ uint64_t pair(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpair(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ uint64_t exp2_pair(uint64_t x)
{
    float a, b;
    unpair(x, a, b);
    return pair(tc_ex2(a), tc_ex2(b));
}
__device__ __forceinline__ float sum_pairs(const uint64_t (&s)[4])
{
    float a, b;
    unpair(add2(add2(s[0], s[1]), add2(s[2], s[3])), a, b);
    return a + b;
}
// N scores of a key (one per query row): adds 2^(score + c[row])
template <int N> __device__ __forceinline__ void key_part(const float (&v)[N], uint64_t sc2, const float* c, uint64_t (&acc)[4])
{
#pragma unroll
    for (int j = 0; j < N; j += 4) {
        const ulonglong2 cc = *reinterpret_cast<const ulonglong2*>(c + j);           // same address for all threads
        acc[(j >> 1) & 3] = add2(acc[(j >> 1) & 3], exp2_pair(fma2(pair(v[j], v[j + 1]), sc2, cc.x)));
        acc[((j >> 1) + 1) & 3] = add2(acc[((j >> 1) + 1) & 3], exp2_pair(fma2(pair(v[j + 2], v[j + 3]), sc2, cc.y)));
    }
}

template <int PASS, int kBlocks>
__global__ void __launch_bounds__(tc_threads(kBlocks), kBlocks == 1 ? 2 : 1) evict_scores_tc_kernel(const EvictTcArgs A, const __grid_constant__ CUtensorMap key_map)
{
    // Pass 2 follows pass 1 on the stream, and what pass 1 waited for is complete (see grid_release): it reads queries,
    // keys and lengths while pass 1 drains, and waits before it reads pass 1's row statistics.
    if (PASS == 1) grid_wait();
    constexpr int kRows = kBlocks * 128, kThreads = tc_threads(kBlocks), kBufs = tc_bufs(kBlocks);
    constexpr unsigned kTileBytes = kTcTile * 256u;
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    __shared__ __align__(8) uint64_t key_full[kBufs], acc_full[2], acc_free[2], vote_full[kBlocks == 2 && PASS == 2 ? 16 : 1];
    __shared__ unsigned tmem_base_s;
    __shared__ int abort_s;
    __shared__ float2 half_ml[kBlocks][128];                // pass 1: row statistics of the second half of the warpgroups
    __shared__ float half_vote[kBlocks == 2 && PASS == 2 ? 2 : 1][2][128];      // pass 2, two row blocks: the second one's share of a tile's votes
    __shared__ __align__(16) float row_c[kRows];            // pass 2: minus the log2-domain softmax offset of each query row

    const int part = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int S = min(A.seq_lens[b], A.S_max);
    if (S <= A.budget) {
        if (PASS == 2) grid_wait();                         // (a grid that ends must have waited)
        return;
    }
    const int G = A.Hq / A.Hkv, R = G * A.W, P = S - A.W;
    const int unit = b * A.Hkv + h;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tl = tid & 127;
    const int wg = warp >> 2, mb = kBlocks == 2 ? wg & 1 : 0, turn = kBlocks == 2 ? wg >> 1 : wg;     // row block; every second tile from `turn` on
    const int tile0 = part * A.tiles_per_cta;
    const int n_tiles_total = (S + kTcTile - 1) / kTcTile;
    const int tile1 = min(n_tiles_total, tile0 + A.tiles_per_cta);
    const int n_tiles = tile1 > tile0 ? tile1 - tile0 : 0;
    // The tile that the sequence ends in comes first (its rows past the end must not be read, so it is staged by hand);
    // pass 1 goes on upwards, pass 2 downwards: it meets first what pass 1 read last, part of which the L2 still holds.
    const bool ragged = n_tiles > 0 && tile1 == n_tiles_total && S % kTcTile != 0;
    auto tile_at = [&](int i) { return PASS == 2 ? tile1 - 1 - i : (ragged ? (i == 0 ? tile1 - 1 : tile0 + i - 1) : tile0 + i); };
    // scores are kept in the log2 domain: 2^(s * log2 e) = e^s, one ex2 per probability
    const float scale = rsqrtf(static_cast<float>(kHeadDim)) * 1.4426950408889634f;

    // operand tiles start on a 1024-byte boundary (the swizzle atom); the launch reserves the slack
    unsigned char* q_s = tc_smem + ((1024u - (tc_smem_u32(tc_smem) & 1023u)) & 1023u);   // [2][kRows][128 B]
    unsigned char* k_s = q_s + kRows * 256;                                                // kBufs x [2][128][128 B]
    const unsigned q_u = tc_smem_u32(q_s), k_u0 = tc_smem_u32(k_s);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&tmem_base_s)), "r"(2 * kRows) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    auto load_tile = [&](int i) {                          // tile i of this CTA into its buffer (one thread)
        const unsigned bar = tc_smem_u32(&key_full[i % kBufs]), dst = k_u0 + static_cast<unsigned>(i % kBufs) * kTileBytes;
        const int t = tile_at(i) * kTcTile;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kTileBytes) : "memory");
        tc_load_keys(dst, &key_map, 0, t, h * A.head_step, b * A.seq_step, bar);
        tc_load_keys(dst + kTcTile * 128u, &key_map, 64, t, h * A.head_step, b * A.seq_step, bar);
    };
    if (tid == kThreads - 32) {
        abort_s = 0;
        for (int i = 0; i < kBufs; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&key_full[i])));
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&acc_full[i])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem_u32(&acc_free[i])), "r"(4 * kBlocks));
        }
        if (kBlocks == 2 && PASS == 2)
            for (int i = 0; i < 16; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&vote_full[i])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int i = ragged ? 1 : 0; i < min(kBufs, n_tiles); ++i) load_tile(i);
    }
    // query rows of the group: row = g*W + w  ->  q_win[b][h*G+g][w][:]  (contiguous over (g, w))
    tc_stage_rows(q_s, kRows, static_cast<const unsigned short*>(A.q_win) + (static_cast<int64_t>(b) * A.Hq + h * G) * A.W * kHeadDim,
                  kHeadDim, R, tid, kThreads);
    if (ragged)
        tc_stage_rows(k_s, kTcTile, static_cast<const unsigned short*>(A.k) + static_cast<int64_t>(b) * A.sb + static_cast<int64_t>(h) * A.sh +
                      static_cast<int64_t>(tile1 - 1) * kTcTile * A.st, A.st, S - (tile1 - 1) * kTcTile, tid, kThreads);
    if (PASS == 2) {                                       // p = 2^(s - c), c = row max + log2(row sum); padding rows give 0
        grid_wait();
        if (tid < kRows) {
            const int r = tid;
            float M = -INFINITY, sum = 0.f;
            if (r < R) {
                const float2* src = reinterpret_cast<const float2*>(A.partial) + static_cast<int64_t>(unit) * A.parts * R + r;
#pragma unroll 8
                for (int p = 0; p < A.parts; ++p) M = fmaxf(M, src[static_cast<int64_t>(p) * R].x);
#pragma unroll 8
                for (int p = 0; p < A.parts; ++p) {
                    const float2 ml = src[static_cast<int64_t>(p) * R];
                    sum += ml.x == -INFINITY ? 0.f : ml.y * exp2f(ml.x - M);
                }
            }
            row_c[r] = (r < R) ? -(M + log2f(sum)) : -INFINITY;
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");          // generic-proxy writes -> tensor-core reads
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    grid_release();                                        // after the tensor-memory allocation: the next kernel's CTAs allocate too
    const unsigned tmem = tmem_base_s;

    float run_m = -INFINITY, run_l = 0.f;                  // pass 1: row 128 mb + tl over this warpgroup's tiles
    if (warp == kThreads / 32 - 1) {
        // ---- one thread feeds the tensor cores: tile i is multiplied into accumulator i & 1 as soon as its keys are there and
        //      the accumulator has been read, and tile i + kBufs is loaded into its buffer as soon as it has been multiplied ----
        if (lane == 0) {
            int loaded = min(kBufs, n_tiles), issued = 0;
            bool ok = true;
            for (int i = 0; i < n_tiles && ok; ++i) {
                if (!(ragged && i == 0)) ok = tc_wait(tc_smem_u32(&key_full[i % kBufs]), ((i / kBufs) & 1) ^ (ragged && i % kBufs == 0 ? 1 : 0), &abort_s);
                if (ok && i >= 2) ok = tc_wait(tc_smem_u32(&acc_free[i & 1]), ((i >> 1) - 1) & 1, &abort_s);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const unsigned k_u = k_u0 + static_cast<unsigned>(i % kBufs) * kTileBytes, d = tmem + static_cast<unsigned>(i & 1) * kRows;
                if (PASS == 1) {
                    constexpr unsigned idesc = tc_idesc(128, kTcTile);
#pragma unroll
                    for (int m = 0; m < kBlocks; ++m)
#pragma unroll
                        for (int k16 = 0; k16 < 8; ++k16) {
                            const unsigned koff = (k16 >> 2) * 128u * 128u + (k16 & 3) * 32u;     // 64-channel block, 32 B per k-step
                            tc_mma(d + m * 128, tc_desc(q_u + (k16 >> 2) * (kRows * 128u) + m * (128u * 128u) + (k16 & 3) * 32u),
                                   tc_desc(k_u + koff), idesc, k16 > 0);
                        }
                } else {
                    constexpr unsigned idesc = tc_idesc(128, kRows);      // padding rows are zero: their scores are finite and row_c drops them
#pragma unroll
                    for (int k16 = 0; k16 < 8; ++k16)
                        tc_mma(d, tc_desc(k_u + (k16 >> 2) * 128u * 128u + (k16 & 3) * 32u),
                               tc_desc(q_u + (k16 >> 2) * (kRows * 128u) + (k16 & 3) * 32u), idesc, k16 > 0);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_u32(&acc_full[i & 1])) : "memory");
                issued = i + 1;
                if (i + kBufs < n_tiles) {
                    ok = tc_wait(tc_smem_u32(&acc_full[i & 1]), (i >> 1) & 1, &abort_s);
                    if (ok) { load_tile(i + kBufs); loaded = i + kBufs + 1; }
                }
            }
            if (!ok) {
                // what is in flight gets one more bounded chance to land before its memory is given up
                record_error(A.status, SPARK_ERR_DEVICE_TIMEOUT);
                volatile int no_abort = 0;
                for (int i = max(issued, ragged ? 1 : 0); i < loaded; ++i)
                    tc_wait(tc_smem_u32(&key_full[i % kBufs]), ((i / kBufs) & 1) ^ (ragged && i % kBufs == 0 ? 1 : 0), &no_abort);
                for (int i = max(0, issued - 2); i < issued; ++i) tc_wait(tc_smem_u32(&acc_full[i & 1]), (i >> 1) & 1, &no_abort);
            }
        }
    } else {
        // ---- epilogue: a thread owns a lane of the accumulator (a query row in pass 1, a key in pass 2) of every second tile ----
        const uint64_t sc2 = pair(scale, scale);
        const int row = mb * 128 + tl;
        const bool row_ok = row < R;
        const int last = P + (row_ok ? row % A.W : 0);
        for (int i = turn; i < n_tiles; i += 2) {
            const int t0 = tile_at(i) * kTcTile;
            if (!__all_sync(0xffffffffu, tc_wait(tc_smem_u32(&acc_full[i & 1]), (i >> 1) & 1, &abort_s))) {
                if (lane == 0) { abort_s = 1; record_error(A.status, SPARK_ERR_DEVICE_TIMEOUT); }
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned acc_u = tmem + static_cast<unsigned>(i & 1) * kRows + mb * 128 + (static_cast<unsigned>((warp & 3) * 32) << 16);
            auto release = [&]() {                         // behind the last read of the accumulator
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem_u32(&acc_free[i & 1])) : "memory");
            };
            if (PASS == 1) {
                if (mb * 128 + (warp & 3) * 32 >= R) { release(); continue; }      // a warp without query rows
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const int tc = t0 + 64 * half;
                    float v[64];
                    tc_ld64(acc_u + 64 * half, v);
                    if (half) release();
                    if (tc + 64 <= P + 1) {                    // every key is visible to every window row
                        float c4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                        for (int j = 4; j < 64; j += 2) c4[(j >> 1) & 3] = max3(c4[(j >> 1) & 3], v[j], v[j + 1]);
                        const float mn = fmaxf(run_m, fmaxf(fmaxf(c4[0], c4[1]), fmaxf(c4[2], c4[3])) * scale);
                        const uint64_t mn2 = pair(-mn, -mn);
                        uint64_t add[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                        for (int j = 0; j < 64; j += 2)
                            add[(j >> 1) & 3] = add2(add[(j >> 1) & 3], exp2_pair(fma2(pair(v[j], v[j + 1]), sc2, mn2)));
                        run_l = run_l * tc_ex2(run_m - mn) + sum_pairs(add);
                        run_m = mn;
                    } else {
                        float cm = -INFINITY;
#pragma unroll
                        for (int j = 0; j < 64; ++j) {
                            const int t = tc + j;
                            v[j] = (row_ok && t <= last && t < S) ? v[j] * scale : -INFINITY;
                            cm = fmaxf(cm, v[j]);
                        }
                        if (cm > -INFINITY) {
                            const float mn = fmaxf(run_m, cm);
                            float add[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                            for (int j = 0; j < 64; ++j) add[j & 3] += tc_ex2(v[j] - mn);    // 2^(-inf) = 0 for masked keys
                            run_l = run_l * tc_ex2(run_m - mn) + ((add[0] + add[1]) + (add[2] + add[3]));
                            run_m = mn;
                        }
                    }
                }
            } else {
                // votes over this warpgroup's 128 query rows: one row block 64 and 64 (added last), two blocks 128 each
                const int n_rows = min(R - mb * 128, 128);
                float vote = 0.f;
                uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
                for (int c0 = 0; c0 < n_rows; c0 += 64) {
                    if (c0 + 32 < n_rows) {
                        float v[64];
                        tc_ld64(acc_u + c0, v);
                        if (c0 + 64 >= n_rows) release();
                        key_part(v, sc2, row_c + mb * 128 + c0, acc);
                    } else {                                   // (padding rows add nothing)
                        float v[32];
                        tc_ld32(acc_u + c0, v);
                        release();
                        key_part(v, sc2, row_c + mb * 128 + c0, acc);
                    }
                    if (kBlocks == 1) {
                        vote += sum_pairs(acc);
                        acc[0] = acc[1] = acc[2] = acc[3] = 0ull;
                    }
                }
                if (kBlocks == 2) vote = sum_pairs(acc);
                if (kBlocks == 2) {
                    // The second row block's warp leaves its share to the first's of the same lane quarter.  (Two slots in turn: it
                    // gets to a slot again only behind the first one's release of the accumulator in between.)
                    const int slot = (i >> 1) & 1;
                    const unsigned bar = tc_smem_u32(&vote_full[(turn * 4 + (warp & 3)) * 2 + slot]);
                    if (mb == 1) {
                        half_vote[turn][slot][tl] = vote;
                        __syncwarp();
                        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
                    } else {
                        if (!__all_sync(0xffffffffu, tc_wait(bar, (i >> 2) & 1, &abort_s))) {
                            if (lane == 0) { abort_s = 1; record_error(A.status, SPARK_ERR_DEVICE_TIMEOUT); }
                            break;
                        }
                        vote += half_vote[turn][slot][tl];
                    }
                }
                if (mb == 0 && t0 + tl < S) A.votes[static_cast<int64_t>(unit) * A.S_max + t0 + tl] = (t0 + tl < P) ? vote : 0.f;
            }
        }
        if (PASS == 1 && turn == 1) half_ml[mb][tl] = make_float2(run_m, run_l);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (PASS == 1 && warp < 4 * kBlocks && mb * 128 + tl < R) {            // the warpgroups with turn 0
        const float2 o = half_ml[mb][tl];
        const float m = fmaxf(run_m, o.x);
        const float l = m == -INFINITY ? 0.f : run_l * tc_ex2(run_m - m) + o.y * tc_ex2(o.x - m);
        const bool have = n_tiles > 0 && !abort_s;
        *reinterpret_cast<float2*>(A.partial + ((static_cast<int64_t>(unit) * A.parts + part) * R + mb * 128 + tl) * 2) =
            make_float2(have ? m : -INFINITY, have ? l : 0.f);
    }
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kRows) : "memory");
    }
}

bool evict_tc_supported(const spark_params& p)
{
    const int R = (p.n_q_heads / p.n_kv_heads) * p.window;
    return p.dtype == SPARK_BF16 && R <= 256;
}

// Tensor map of the keys: (channel, token, head, sequence), copied in blocks of 64 channels x 128 tokens.  The kernels copy
// only blocks whose rows all lie inside their sequence, so the token extent is only a bound.  False where the driver makes none: a
// stride of 2^40 bytes or more, or a driver that wants ascending strides (the heads of token-major keys lie closer than the tokens).
static bool key_tensor_map(CUtensorMap* map, EvictTcArgs& A, const spark_params& p, int dev)
{
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {                      // looked up once
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<Encode>(f);
    }();
    if (!encode) return false;
    // heads or sequences that share their keys (stride 0) are one coordinate
    A.head_step = p.n_kv_heads > 1 && A.sh > 0 ? 1 : 0;
    A.seq_step = p.batch > 1 && A.sb > 0 ? 1 : 0;
    const cuuint64_t dims[4] = {kHeadDim, static_cast<cuuint64_t>(A.S_max), A.head_step ? static_cast<cuuint64_t>(p.n_kv_heads) : 1u,
                                A.seq_step ? static_cast<cuuint64_t>(p.batch) : 1u};
    const cuuint64_t row = static_cast<cuuint64_t>(A.st) * 2;
    const cuuint64_t strides[3] = {row, A.head_step ? static_cast<cuuint64_t>(A.sh) * 2 : row, A.seq_step ? static_cast<cuuint64_t>(A.sb) * 2 : row};
    const cuuint32_t box[4] = {64, kTcTile, 1, 1}, ones[4] = {1, 1, 1, 1};
    auto make = [&]() {
        return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(A.k), dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    // a thread that has made no runtime call yet has no context, which this driver call wants: binding the current device gives it one
    return make() || (cudaSetDevice(dev) == cudaSuccess && make());
}

// Tensor-core votes: the workspace regions `partial` and `votes` of the CUDA-core path (row statistics stay on chip).  `done` says
// whether they were enqueued: where the keys have no tensor map they are not, and nothing is.
spark_status launch_evict_votes_tc(const spark_params& p, const void* q_win, const void* k, int64_t sb, int64_t sh,
                                   int64_t st, const int32_t* seq_lens, int32_t max_seq_tokens, float* partial,
                                   float* votes, int* status, cudaStream_t stream, int* launches, bool* done)
{
    const int R = (p.n_q_heads / p.n_kv_heads) * p.window;
    const int Rpad = (R + 127) / 128 * 128;
    EvictTcArgs A;
    A.q_win = q_win; A.k = k; A.sb = sb; A.sh = sh; A.st = st; A.seq_lens = seq_lens;
    A.Hq = p.n_q_heads; A.Hkv = p.n_kv_heads; A.W = p.window; A.budget = p.token_budget; A.S_max = max_seq_tokens;
    const int n_tiles = (max_seq_tokens + kTcTile - 1) / kTcTile;
    // A CTA pays a fixed start-up (tensor-memory allocation, the query block, the first key tile), so the tiles are cut into
    // one wave of CTAs, at least 8 tiles each.  Up to 128 query rows two CTAs are resident per SM; above that one takes 193 KB
    // of shared memory and all 512 tensor-memory columns.  (us per evicting prefill with 129 to 256 rows, cut for two CTAs per
    // SM -> for one: 1 x 131072 with 28 / 4 heads 188 -> 169, with 64 / 8 heads 308 -> 296, 2 x 20000 102 -> 72.)
    int dev = 0;
    DeviceInfo info;
    if (!device_info(&dev, &info)) return SPARK_ERR_CUDA;
    const int64_t units = static_cast<int64_t>(p.batch) * p.n_kv_heads;
    const int64_t wave = (Rpad <= 128 ? 2 : 1) * static_cast<int64_t>(info.n_sms);
    const int64_t parts = units < wave ? wave / units : 1;
    int64_t per = (n_tiles + parts - 1) / parts;
    if (per < 8) per = 8;
    if (per > n_tiles) per = n_tiles > 0 ? n_tiles : 1;
    A.tiles_per_cta = static_cast<int>(per);
    A.parts = (n_tiles + A.tiles_per_cta - 1) / A.tiles_per_cta;
    A.partial = partial; A.votes = votes; A.status = status;
    CUtensorMap key_map;
    *done = key_tensor_map(&key_map, A, p, dev);
    if (!*done) return SPARK_OK;
    static unsigned char smem_raised[4][kMaxDevices] = {};
    auto both = [&](auto blocks) {
        constexpr int kBlocks = decltype(blocks)::value;
        const size_t smem = kBlocks * 128 * 256 + tc_bufs(kBlocks) * kTcTile * 256 + 1024;     // queries, key buffers, alignment slack
        if (!allow_max_smem(evict_scores_tc_kernel<1, kBlocks>, dev, info.smem_optin, smem_raised[2 * kBlocks - 2]) ||
            !allow_max_smem(evict_scores_tc_kernel<2, kBlocks>, dev, info.smem_optin, smem_raised[2 * kBlocks - 1]))
            return false;
        const dim3 grid(A.parts, p.n_kv_heads, p.batch);
        launch_kernel(evict_scores_tc_kernel<1, kBlocks>, grid, dim3(tc_threads(kBlocks)), smem, stream, A, key_map);
        launch_kernel(evict_scores_tc_kernel<2, kBlocks>, grid, dim3(tc_threads(kBlocks)), smem, stream, A, key_map);
        return true;
    };
    if (!(Rpad <= 128 ? both(std::integral_constant<int, 1>()) : both(std::integral_constant<int, 2>()))) return SPARK_ERR_CUDA;
    *launches += 2;
    return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace spark
