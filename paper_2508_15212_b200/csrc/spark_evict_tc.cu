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
// Tiles are pipelined two deep: the epilogue of tile i (bound by its exponentials, 1024 cycles of the SM's special
// function units per 128 x 128 scores) runs under the MMAs of tile i + 1 and the loads of tile i + 2.  With load, MMA and
// epilogue in turn, one warpgroup and scalar fp32 the two passes over 8 x 131072 keys took 81 + 69 us and 8 us of
// row statistics between them, now 66 + 63 us.
// Operands are staged in shared memory by ordinary loads in the canonical K-major 128-byte-swizzled
// layout that the matrix descriptors name (row r of a 64-channel block at r*128 bytes, its 16-byte
// chunks XOR-ed with r & 7; 8-row groups 1024 bytes apart).  One thread issues the MMAs; completion
// arrives on an mbarrier through tcgen05.commit; every wait is bounded.
#include "spark_common.cuh"

namespace spark {

constexpr int kTcTile = 128;            // keys per tile
constexpr int kTcThreads = 256;         // two warpgroups share a tile's epilogue (a tensor-memory lane is readable by both)
constexpr unsigned kTcSpin = 1u << 22;

struct EvictTcArgs {
    const void* q_win;
    const void* k;
    int64_t sb, sh, st;
    const int32_t* seq_lens;
    int Hq, Hkv, W, budget;
    int S_max, tiles_per_cta, parts;     // parts = CTAs per unit
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
__device__ __forceinline__ unsigned tc_idesc(int M, int N)
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
                                              int valid, int tid)
{
    for (int i = tid; i < rows_alloc * 16; i += kTcThreads) {
        const int r = i >> 4, ch16 = i & 15;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < valid) v = *reinterpret_cast<const uint4*>(src + static_cast<int64_t>(r) * stride + ch16 * 8);
        const int kb = ch16 >> 3, c8 = ch16 & 7;
        *reinterpret_cast<uint4*>(dst + static_cast<size_t>(kb) * rows_alloc * 128 + r * 128 + ((c8 ^ (r & 7)) << 4)) = v;
    }
}

// The same copy for a tile of 128 keys with 16-byte asynchronous copies (rows >= valid are zero-filled).  A thread
// copies the same 16-byte chunk of every sixteenth row (so the swizzle term is constant): a pointer increment and a copy per row.
__device__ __forceinline__ void tc_stage_keys_async(unsigned dst_u, const unsigned short* src, int64_t stride, int valid, int tid)
{
    constexpr int kRows = kTcThreads / 16;
    const int r0 = tid >> 4, ch16 = tid & 15;
    const unsigned d = dst_u + static_cast<unsigned>(ch16 >> 3) * (kTcTile * 128u) + r0 * 128u + (((ch16 & 7) ^ (r0 & 7)) << 4);
    const unsigned short* g = src + static_cast<int64_t>(r0) * stride + ch16 * 8;
    const int64_t step = kRows * stride;
    if (valid >= kTcTile) {
#pragma unroll
        for (int i = 0; i < kTcTile / kRows; ++i) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + i * (kRows * 128u)), "l"(g) : "memory");
            g += step;
        }
    } else {
#pragma unroll 1
        for (int i = 0; i < kTcTile / kRows; ++i) {
            const bool live = r0 + kRows * i < valid;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + i * (kRows * 128u)), "l"(live ? g : src), "r"(live ? 16 : 0) : "memory");
            g += step;
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
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

template <int PASS>
__global__ void __launch_bounds__(kTcThreads, 2) evict_scores_tc_kernel(EvictTcArgs A)
{
    // Pass 2 follows pass 1 on the stream, and what pass 1 waited for is complete (see grid_release): it reads queries,
    // keys and lengths while pass 1 drains, and waits before it reads pass 1's row statistics.
    if (PASS == 1) grid_wait();
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    __shared__ __align__(8) uint64_t mma_bar;
    __shared__ unsigned tmem_base_s;
    __shared__ float2 half_ml[2][128];                      // pass 1: the second warpgroup's row statistics
    __shared__ float half_vote[2][128];                     // pass 2: its votes of the last two tiles
    __shared__ __align__(16) float row_c[256];              // pass 2: minus the log2-domain softmax offset of each query row

    const int part = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int S = min(A.seq_lens[b], A.S_max);
    if (S <= A.budget) {
        if (PASS == 2) grid_wait();                         // (a grid that ends must have waited)
        return;
    }
    const int G = A.Hq / A.Hkv, R = G * A.W, P = S - A.W;
    const int Rpad = (R + 127) / 128 * 128;                   // staged query rows (1 or 2 blocks of 128)
    const int unit = b * A.Hkv + h;
    const int tid = threadIdx.x, warp = tid >> 5, wg = tid >> 7, tl = tid & 127;      // warpgroup, tensor-memory lane
    const int tile0 = part * A.tiles_per_cta;
    const int n_tiles_total = (S + kTcTile - 1) / kTcTile;
    const int tile1 = min(n_tiles_total, tile0 + A.tiles_per_cta);
    // scores are kept in the log2 domain: 2^(s * log2 e) = e^s, one ex2 per probability
    const float scale = rsqrtf(static_cast<float>(kHeadDim)) * 1.4426950408889634f;

    // operand tiles start on a 1024-byte boundary (the swizzle atom); the launch reserves the slack
    unsigned char* q_s = tc_smem + ((1024u - (tc_smem_u32(tc_smem) & 1023u)) & 1023u);   // [2][Rpad][128 B]
    unsigned char* k_s = q_s + static_cast<size_t>(Rpad) * 256;                            // 2 buffers of [2][128][128 B]
    const int n_cols = Rpad;                                  // tensor-memory columns of one accumulator stage: 128 or 256

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&tmem_base_s)), "r"(2 * n_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&mma_bar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // query rows of the group: row = g*W + w  ->  q_win[b][h*G+g][w][:]  (contiguous over (g, w))
    tc_stage_rows(q_s, Rpad, static_cast<const unsigned short*>(A.q_win) + (static_cast<int64_t>(b) * A.Hq + h * G) * A.W * kHeadDim,
                  kHeadDim, R, tid);
    const unsigned q_u = tc_smem_u32(q_s), k_u0 = tc_smem_u32(k_s);
    const unsigned short* k_unit = static_cast<const unsigned short*>(A.k) + static_cast<int64_t>(b) * A.sb +
                                   static_cast<int64_t>(h) * A.sh;
    const int n_tiles = tile1 > tile0 ? tile1 - tile0 : 0;
    auto stage_keys = [&](int i) {                         // key tile i of this CTA into buffer i & 1
        const int t = (tile0 + i) * kTcTile;
        tc_stage_keys_async(k_u0 + static_cast<unsigned>(i & 1) * (kTcTile * 256u), k_unit + static_cast<int64_t>(t) * A.st,
                            A.st, min(kTcTile, S - t), tid);
    };
    if (n_tiles > 0) stage_keys(0);
    if (PASS == 2) {                                       // p = 2^(s - c), c = row max + log2(row sum); padding rows give 0
        grid_wait();
        for (int r = tid; r < 256; r += kTcThreads) {
            float M = -INFINITY, sum = 0.f;
            if (r < R) {
                const float2* src = reinterpret_cast<const float2*>(A.partial) + static_cast<int64_t>(unit) * A.parts * R + r;
                for (int p = 0; p < A.parts; ++p) M = fmaxf(M, src[static_cast<int64_t>(p) * R].x);
                for (int p = 0; p < A.parts; ++p) {
                    const float2 ml = src[static_cast<int64_t>(p) * R];
                    sum += ml.x == -INFINITY ? 0.f : ml.y * exp2f(ml.x - M);
                }
            }
            row_c[r] = (r < R) ? -(M + log2f(sum)) : -INFINITY;
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");          // generic-proxy writes -> tensor-core reads
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    grid_release();                                        // after the tensor-memory allocation: the next kernel's CTAs allocate too
    const unsigned tmem = tmem_base_s;
    // all MMAs of key tile i into accumulator stage i & 1 (one thread)
    auto issue_mma = [&](int i) {
        const unsigned k_u = k_u0 + static_cast<unsigned>(i & 1) * (kTcTile * 256u), d = tmem + static_cast<unsigned>(i & 1) * n_cols;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (PASS == 1) {
            const unsigned idesc = tc_idesc(128, kTcTile);
            for (int mb = 0; mb < Rpad / 128; ++mb)
#pragma unroll
                for (int k16 = 0; k16 < 8; ++k16) {
                    const unsigned koff = (k16 >> 2) * 128u * 128u + (k16 & 3) * 32u;     // 64-channel block, 32 B per k-step
                    tc_mma(d + mb * 128, tc_desc(q_u + (k16 >> 2) * (Rpad * 128u) + mb * (128u * 128u) + (k16 & 3) * 32u),
                           tc_desc(k_u + koff), idesc, k16 > 0);
                }
        } else {
            const unsigned idesc = tc_idesc(128, Rpad);    // padding rows are zero: their scores are finite and row_c drops them
#pragma unroll
            for (int k16 = 0; k16 < 8; ++k16)
                tc_mma(d, tc_desc(k_u + (k16 >> 2) * 128u * 128u + (k16 & 3) * 32u),
                       tc_desc(q_u + (k16 >> 2) * (Rpad * 128u) + (k16 & 3) * 32u), idesc, k16 > 0);
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem_u32(&mma_bar)) : "memory");
    };
    if (tid == 0 && n_tiles > 0) issue_mma(0);
    if (n_tiles > 1) stage_keys(1);

    float run_m[2] = {-INFINITY, -INFINITY}, run_l[2] = {0.f, 0.f};       // pass 1: rows tl and 128 + tl, this warpgroup's columns
    float prev_vote = 0.f;                                 // pass 2: first warpgroup, the tile before
    bool dead = false;
    const uint64_t sc2 = pair(scale, scale);
    auto write_vote = [&](int t, float vote) {
        if (t < S) A.votes[static_cast<int64_t>(unit) * A.S_max + t] = (t < P) ? vote : 0.f;
    };

    // Tile i's epilogue runs while tile i + 1 is multiplied (the other accumulator stage) and tile i + 2 is loaded (the key
    // buffer that tile i's MMAs have released); one CTA barrier per tile.
    for (int i = 0; i < n_tiles; ++i) {
        const int t0 = (tile0 + i) * kTcTile;
        asm volatile("cp.async.wait_group 0;" ::: "memory");             // this thread's part of tile i + 1 has landed
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // wait for the MMAs of tile i (bounded).  The verdict is made CTA-uniform by the barrier, so that the
        // warp-collective tensor-memory loads of the epilogue are never executed divergently and, once a wait has
        // run out, no thread issues further MMAs or reads the accumulator.
        unsigned ok = 0u;
        for (unsigned it = 0; it < kTcSpin && !ok; ++it)
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(ok) : "r"(tc_smem_u32(&mma_bar)), "r"(i & 1) : "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); // the previous epilogue's reads of the other stage
        dead = __syncthreads_or(!ok) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (dead) {
            if (tid == 0) record_error(A.status, SPARK_ERR_DEVICE_TIMEOUT);
            // give the MMAs that were issued one more bounded chance to retire before the accumulator is freed
            for (unsigned it = 0; it < kTcSpin && !ok; ++it)
                asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                             : "=r"(ok) : "r"(tc_smem_u32(&mma_bar)), "r"(i & 1) : "memory");
            break;
        }
        if (tid == 0 && i + 1 < n_tiles) issue_mma(i + 1);
        if (i + 2 < n_tiles) stage_keys(i + 2);
        const unsigned lane_addr = tmem + static_cast<unsigned>(i & 1) * n_cols + (static_cast<unsigned>((warp & 3) * 32) << 16);
        if (PASS == 1) {
            for (int mb = 0; mb < Rpad / 128; ++mb) {
                if (mb * 128 + (warp & 3) * 32 >= R) continue;           // a warp without query rows
                const int row = mb * 128 + tl, tc = t0 + 64 * wg;        // this warpgroup's 64 keys
                const bool row_ok = row < R;
                const int last = P + (row_ok ? row % A.W : 0);
                float m = run_m[mb], l = run_l[mb];
                float v[64];
                tc_ld64(lane_addr + mb * 128 + 64 * wg, v);
                if (tc + 64 <= P + 1) {                        // every key is visible to every window row
                    float c4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
                    for (int j = 4; j < 64; j += 2) c4[(j >> 1) & 3] = max3(c4[(j >> 1) & 3], v[j], v[j + 1]);
                    const float mn = fmaxf(m, fmaxf(fmaxf(c4[0], c4[1]), fmaxf(c4[2], c4[3])) * scale);
                    const uint64_t mn2 = pair(-mn, -mn);
                    uint64_t add[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                    for (int j = 0; j < 64; j += 2)
                        add[(j >> 1) & 3] = add2(add[(j >> 1) & 3], exp2_pair(fma2(pair(v[j], v[j + 1]), sc2, mn2)));
                    l = l * tc_ex2(m - mn) + sum_pairs(add);
                    m = mn;
                } else {
                    float cm = -INFINITY;
#pragma unroll
                    for (int j = 0; j < 64; ++j) {
                        const int t = tc + j;
                        v[j] = (row_ok && t <= last && t < S) ? v[j] * scale : -INFINITY;
                        cm = fmaxf(cm, v[j]);
                    }
                    if (cm > -INFINITY) {
                        const float mn = fmaxf(m, cm);
                        float add[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int j = 0; j < 64; ++j) add[j & 3] += tc_ex2(v[j] - mn);    // 2^(-inf) = 0 for masked keys
                        l = l * tc_ex2(m - mn) + ((add[0] + add[1]) + (add[2] + add[3]));
                        m = mn;
                    }
                }
                run_m[mb] = m; run_l[mb] = l;
            }
        } else {
            // this warpgroup's half of the query rows (padding rows add nothing)
            const int c1 = min(R, (wg + 1) * (Rpad / 2));
            uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
            int c0 = wg * (Rpad / 2);
#pragma unroll 1
            for (; c0 + 32 < c1; c0 += 64) {
                float v[64];
                tc_ld64(lane_addr + c0, v);
                key_part(v, sc2, row_c + c0, acc);
            }
            if (c0 < c1) {
                float v[32];
                tc_ld32(lane_addr + c0, v);
                key_part(v, sc2, row_c + c0, acc);
            }
            const float vote = sum_pairs(acc);
            // the second warpgroup leaves its share; the first adds it behind the next tile's barrier
            if (wg == 1) half_vote[i & 1][tl] = vote;
            else {
                if (i > 0) write_vote(t0 - kTcTile + tl, prev_vote + half_vote[(i - 1) & 1][tl]);
                prev_vote = vote;
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (PASS == 1 && wg == 1) {
        half_ml[0][tl] = make_float2(run_m[0], run_l[0]);
        half_ml[1][tl] = make_float2(run_m[1], run_l[1]);
    }
    __syncthreads();
    if (PASS == 1 && wg == 0)
        for (int mb = 0; mb < Rpad / 128; ++mb) {
            const int row = mb * 128 + tl;
            if (row < R) {
                const float2 o = half_ml[mb][tl];
                const float m = fmaxf(run_m[mb], o.x);
                const float l = m == -INFINITY ? 0.f : run_l[mb] * tc_ex2(run_m[mb] - m) + o.y * tc_ex2(o.x - m);
                const bool have = n_tiles > 0 && !dead;
                *reinterpret_cast<float2*>(A.partial + ((static_cast<int64_t>(unit) * A.parts + part) * R + row) * 2) =
                    make_float2(have ? m : -INFINITY, have ? l : 0.f);
            }
        }
    if (PASS == 2 && wg == 0 && n_tiles > 0 && !dead)
        write_vote((tile0 + n_tiles - 1) * kTcTile + tl, prev_vote + half_vote[(n_tiles - 1) & 1][tl]);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * n_cols) : "memory");
}

bool evict_tc_supported(const spark_params& p)
{
    const int R = (p.n_q_heads / p.n_kv_heads) * p.window;
    return p.dtype == SPARK_BF16 && R <= 256;
}

// Tensor-core votes: the workspace regions `partial` and `votes` of the CUDA-core path (row statistics stay on chip).
spark_status launch_evict_votes_tc(const spark_params& p, const void* q_win, const void* k, int64_t sb, int64_t sh,
                                   int64_t st, const int32_t* seq_lens, int32_t max_seq_tokens, float* partial,
                                   float* votes, int* status, cudaStream_t stream, int* launches)
{
    const int R = (p.n_q_heads / p.n_kv_heads) * p.window;
    const int Rpad = (R + 127) / 128 * 128;
    EvictTcArgs A;
    A.q_win = q_win; A.k = k; A.sb = sb; A.sh = sh; A.st = st; A.seq_lens = seq_lens;
    A.Hq = p.n_q_heads; A.Hkv = p.n_kv_heads; A.W = p.window; A.budget = p.token_budget; A.S_max = max_seq_tokens;
    const int n_tiles = (max_seq_tokens + kTcTile - 1) / kTcTile;
    // A CTA pays a fixed start-up (tensor-memory allocation, the query block, the first key tile), so the tiles are cut into
    // one wave of CTAs, at least 8 tiles each.  Up to 128 query rows two CTAs are resident per SM; above that one takes 129 KB
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
    const size_t smem = static_cast<size_t>(Rpad) * 256 + 2 * kTcTile * 256 + 1024;     // queries, two key buffers, alignment slack
    static unsigned char smem_raised[2][kMaxDevices] = {};
    if (!allow_max_smem(evict_scores_tc_kernel<1>, dev, info.smem_optin, smem_raised[0]) ||
        !allow_max_smem(evict_scores_tc_kernel<2>, dev, info.smem_optin, smem_raised[1]))
        return SPARK_ERR_CUDA;
    const dim3 grid(A.parts, p.n_kv_heads, p.batch);
    launch_kernel(evict_scores_tc_kernel<1>, grid, dim3(kTcThreads), smem, stream, A);
    launch_kernel(evict_scores_tc_kernel<2>, grid, dim3(kTcThreads), smem, stream, A);
    *launches += 2;
    return cudaGetLastError() == cudaSuccess ? SPARK_OK : SPARK_ERR_CUDA;
}

}  // namespace spark
