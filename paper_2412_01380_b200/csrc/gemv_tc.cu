// Batched decode, 3 to 16 tokens, BF16 weights: the sparse product over the UNION of the tokens' kept
// columns (each row read once; token b uses a row only if its own mask keeps it) is a dense
// contraction D[tokens][outputs] += X^T[tokens][rows] W~[rows][outputs], and runs on the fifth-
// generation tensor cores:
//   * a CTA owns a 512-byte segment of the packed rows (256 outputs) and a part of the union's
//     rows; 16 warps stream the rows with 16-byte asynchronous copies (a whole segment per warp
//     instruction; rounds of 64 rows, three rounds in flight in a ring of four buffers) straight
//     into shared memory in the layout that a 128-byte-swizzled
//     MN-major operand descriptor names: the outputs of a row are contiguous, so the weights are the
//     B operand (N = 256) as they arrive, untransposed, and each byte is read by one MMA only;
//   * the tokens' values of the union's rows, zeroed where a token drops the row and split into two bfloat16, are gathered
//     ONCE per product by xt_build_kernel (16 scattered loads per row) into a table of 64 bytes per column.  The loaders copy a
//     row's 64 bytes as the MN-major A operand: row n = the high halves of token n, row 16 + n the low halves, the other rows of
//     the M = 128 tile zero.  (Every CTA gathering its rows' values for itself, four bytes at a time, is what the load path
//     cannot take: 16 tokens' gate/up product 86 us with registers and warps of their own, 105 us with asynchronous copies of four
//     bytes, 60 us like this.  The product's blocks sharing the gathering and waiting for one another saves a launch and is slower
//     all the same (16 tokens at 5120 / 17920, keep ratio 0.25: 122.4 us per step against 116.5; a union of 64 of 8192 columns, one segment:
//     47.6 against 7.9), and where there are more segments than SMs the first blocks wait for some that start after them);
//   * one thread of a seventeenth warp issues one tcgen05.mma (M = 128, N = 256, K = 16) per 16 rows
//     once the loader warps have arrived on the buffer's "full" barrier; the accumulator lives in
//     tensor memory (256 columns) for the whole kernel, and a tcgen05.commit per round tells the
//     loaders through a second mbarrier when a buffer may be overwritten;
//   * four warps read the 32 useful accumulator rows with tcgen05.ld, add the low-half row to the high-half row and leave the
//     sums in shared memory; then all threads apply silu(gate) * up (a 16-column chunk is 8 gate outputs and
//     their 8 up outputs), or send the row part to the last part's CTA, which adds the parts up first.
// All products are exact in binary32 (bf16 x bf16); sums are binary32 in the tensor core's order.
// Every wait on an mbarrier is bounded; on expiry the kernel records a status word, frees its
// tensor memory and leaves.
#include <cuda_bf16.h>

#include "common.cuh"
#include "gemv_common.cuh"

namespace {

constexpr int TC_LOAD_WARPS = 16;                // warps that stream rows, and one that issues the MMAs
constexpr int TC_WARPS = TC_LOAD_WARPS + 1;
constexpr int TC_THREADS = TC_WARPS * 32;
constexpr int TC_U = 4;                          // rows per lane and round
constexpr int TC_ROUND_ROWS = TC_LOAD_WARPS * TC_U;   // 64 rows = 4 K-blocks of 16 per round
constexpr int TC_KB = TC_ROUND_ROWS / 16;
constexpr int TC_BUFS = 4;                       // ring of round buffers: three rounds of copies in flight
constexpr int TC_SEG = 512;                      // bytes of a packed row per CTA: 256 bf16 outputs = N
constexpr int TC_N = 16;                         // tokens
constexpr int TC_A_KB_BYTES = 16 * TC_SEG;       // one K-block of weights: [k group 2][output block 4][8 rows][128 B]
constexpr int TC_B_KB_BYTES = 128 * 16 * 2;      // one K-block of values: [row group 16][k group 2][8 rows][16 B]
constexpr int TC_TMEM_COLS = 256;                // one accumulator: 128 lanes x 256 binary32 columns

// Rows per in-kernel list: a list boundary drains the copy ring, so a part should be one list
// (16 tokens at keep ratio 0.25 keep ~5100 of 5120 gate/up rows, ~2500 down rows per part).
constexpr int TC_LIST_ROWS = 8192;

struct __align__(1024) TcSmem {
    unsigned char a[TC_BUFS][TC_KB * TC_A_KB_BYTES];   // weights, 4 x 32 KB
    unsigned char b[TC_BUFS][TC_KB * TC_B_KB_BYTES];   // token values, 4 x 16 KB
    uint64_t full[TC_BUFS];                      // the loader warps' copies into buffer i have landed
    uint64_t done[TC_BUFS];                      // the MMAs that read buffer i have completed
    uint32_t tmem_base;
    int n_total;
    int fail;
    int wsum[TC_WARPS];
    uint32_t words[DIP_MAX_D / 32];
    int pre[DIP_MAX_D / 32];
    uint16_t idx[TC_LIST_ROWS];
};

// Shared-memory operand descriptor: start address, leading / stride byte offsets (in 16-byte units),
// descriptor version 1, layout type (0 = no swizzle, 2 = 128-byte swizzle).
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout)
{
    return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) | ((uint64_t)(sbo_bytes >> 4) << 32) |
           (1ull << 46) | ((uint64_t)layout << 61);
}

// Instruction descriptor of kind::f16: binary32 accumulate, bfloat16 A and B, A (token values)
// MN-major (token slots contiguous), B (weights) MN-major (outputs contiguous), N = 256, M = 128.
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t accumulate)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(TC_IDESC), "r"(accumulate) : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 64 consecutive columns of this warp's 32 lanes of tensor memory: thread = lane, register = column
// (four 16-column loads in flight, one wait).
__device__ __forceinline__ void tc_ld64(uint32_t taddr, float (&v)[64])
{
    uint32_t r[64];
#pragma unroll
    for (int c = 0; c < 4; ++c)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                     : "=r"(r[16 * c + 0]), "=r"(r[16 * c + 1]), "=r"(r[16 * c + 2]), "=r"(r[16 * c + 3]), "=r"(r[16 * c + 4]),
                       "=r"(r[16 * c + 5]), "=r"(r[16 * c + 6]), "=r"(r[16 * c + 7]), "=r"(r[16 * c + 8]), "=r"(r[16 * c + 9]),
                       "=r"(r[16 * c + 10]), "=r"(r[16 * c + 11]), "=r"(r[16 * c + 12]), "=r"(r[16 * c + 13]),
                       "=r"(r[16 * c + 14]), "=r"(r[16 * c + 15])
                     : "r"(taddr + 16 * c));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}

struct TcParams {
    int n_slabs, nparts;
    const uint16_t *xt;        // [d_in][32] the table: 16 high, 16 low halves
    unsigned long long block_wait_ns;
};

// The tokens' values of every column of the union, ready for the tensor core: xt[i][n] = bfloat16 high
// half of token n's value at column i (zero where the token's own mask drops the column or
// n >= batch), xt[i][16 + n] = the low half; columns outside the union are not written (and never
// read).  Built once per product instead of once per CTA (the values are 16 scattered 4-byte loads
// per column).  A block takes two mask words per pass; 16 consecutive threads are the 16 tokens of
// one column.
__global__ void __launch_bounds__(1024, 1)
xt_build_kernel(const uint32_t *__restrict__ mask_bits, const float *__restrict__ v, int batch, int d_in, int mask_words,
                uint16_t *__restrict__ xt)
{
    const int tid = threadIdx.x;
    const int n = tid & 15, bit = (tid >> 4) & 31, half = tid >> 9;
    dip_grid_dependency_wait();
    dip_launch_dependents();
    for (int w = 2 * blockIdx.x + half; w < mask_words; w += 2 * gridDim.x) {
        const int idx = w * 32 + bit;
        const bool mine = n < batch && idx < d_in && ((mask_bits[(size_t)n * mask_words + w] >> bit) & 1u);
        // in the union if any of the 16 tokens (a half-warp) keeps the column
        const unsigned any = __ballot_sync(0xffffffffu, mine) & (0xffffu << (tid & 16));
        if (!any) continue;
        const float x = mine ? __ldg(v + (size_t)n * d_in + idx) : 0.f;
        const __nv_bfloat16 hi = __float2bfloat16_rn(x);
        const __nv_bfloat16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
        xt[(size_t)idx * 32 + n] = __bfloat16_as_ushort(hi);
        xt[(size_t)idx * 32 + 16 + n] = __bfloat16_as_ushort(lo);
    }
}

template <int WHICH>
__global__ void __launch_bounds__(TC_THREADS, 1)
gemv_tc_kernel(const GemvParams p, const TcParams q)
{
    extern __shared__ unsigned char tc_smem_raw[];
    TcSmem &s = *reinterpret_cast<TcSmem *>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
    DIP_TRACE_MIN(p.tr, 0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slab = (int)blockIdx.x % q.n_slabs, part = (int)blockIdx.x / q.n_slabs, nparts = q.nparts;
    const size_t byte_off = (size_t)slab * TC_SEG + lane * 16;
    const bool lane_ok = byte_off < p.row_bytes;

    // ---- set-up: tensor memory for the two accumulator tiles, the buffers' barriers ----
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s.tmem_base)),
                     "n"(TC_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < TC_BUFS; ++i) {
            mbar_init(&s.full[i], TC_LOAD_WARPS);
            mbar_init(&s.done[i], 1);
        }
        s.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s.tmem_base;
    // the rows of the M = 128 tile that no token uses stay zero
    for (int i = tid; i < (int)(sizeof(s.b) / 16); i += TC_THREADS) reinterpret_cast<uint4 *>(&s.b[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // (the block barriers below order them before any MMA)
    dip_grid_dependency_wait();        // the masks and the vectors come from the previous kernels
    DIP_TRACE_MIN(p.tr, 1);
    dip_launch_dependents();

    // ---- 1. the union of the tokens' mask words (two neighbours per thread) and its popcount prefix ----
    {
        static_assert(2 * TC_THREADS >= DIP_MAX_D / 32, "");
        uint32_t u[2] = {0u, 0u};
#pragma unroll 4
        for (int b = 0; b < p.batch; ++b)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (2 * tid + j < p.mask_words) u[j] |= __ldg(p.mask_bits + (size_t)b * p.mask_words + 2 * tid + j);
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (2 * tid + j == p.mask_words - 1 && (p.d_in & 31)) u[j] &= (1u << (p.d_in & 31)) - 1u;
        const int c = __popc(u[0]) + __popc(u[1]);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int n = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += n;
        }
        if (lane == 31) s.wsum[warp] = incl;
        __syncthreads();
        int pre = (int)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)s.wsum[lane] : 0u) + incl - c;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int w = 2 * tid + j;
            if (w < p.mask_words) {
                s.words[w] = u[j];
                s.pre[w] = pre;
            }
            pre += __popc(u[j]);
        }
        if (tid == TC_THREADS - 1) s.n_total = pre;
    }
    __syncthreads();
    const int n_total = s.n_total;
    const int r_begin = (int)(((long long)part * n_total) / nparts);
    const int r_end = (int)(((long long)(part + 1) * n_total) / nparts);
    const char *base = p.W + byte_off;

    // this lane's place in a round of weights: row slot k = warp of K-block u, 16-byte chunk `lane` of the segment
    const uint32_t a_off = (uint32_t)(((warp & 15) >> 3) * 4096 + (lane >> 3) * 1024 + (warp & 7) * 128 + (((lane & 7) ^ (warp & 7)) << 4));
    // and, of threads 0 .. 4 TC_ROUND_ROWS - 1, of values: row tid / 4 of the round, 16-byte chunk tid % 4 of its 64 bytes in xt
    // (the high halves of tokens 0-7, 8-15, the low halves of tokens 0-7, 8-15) = A rows 8 (tid % 4) .. + 7
    // at that k: core matrices of 8 k x 16 bytes, the 16 row groups 128 B apart, the two k groups 2 KB apart
    const int bb_row = (tid >> 2) & (TC_ROUND_ROWS - 1), bb_mg = tid & 3;
    const uint32_t b_off = (uint32_t)((bb_row >> 4) * TC_B_KB_BYTES + ((bb_row & 15) >> 3) * 2048 + bb_mg * 128 + (bb_row & 7) * 16);

    int g = 0;                         // rounds so far (buffer g & 1)
    bool failed = false;

    // The part's rows go through in lists of at most TC_LIST_ROWS (the in-kernel row list), a list in
    // rounds of TC_ROUND_ROWS.  Warps 0-15 load and store; warp 16 issues the MMAs.
    for (int list_begin = r_begin; list_begin < r_end; list_begin += TC_LIST_ROWS) {
        const int n_rows = min(r_end - list_begin, TC_LIST_ROWS);
        if (list_begin != r_begin) __syncthreads();               // everyone is done with the previous list
        {
            const int lo_rank = list_begin, hi_rank = list_begin + n_rows;
            for (int b = tid; b < 4 * p.mask_words; b += TC_THREADS) {        // a byte of a word
                const int w = b >> 2, low = 8 * (b & 3);
                const uint32_t all = s.words[w];
                uint32_t u = all & (0xffu << low);
                int rank = s.pre[w] + __popc(all & ((1u << low) - 1u));
                if (rank >= hi_rank || rank + __popc(u) <= lo_rank) continue;
                for (; u; u &= u - 1, ++rank)
                    if (rank >= lo_rank && rank < hi_rank) s.idx[rank - lo_rank] = (uint16_t)(w * 32 + __ffs(u) - 1);
            }
        }
        __syncthreads();
        const int n_rounds = (n_rows + TC_ROUND_ROWS - 1) / TC_ROUND_ROWS;

        if (warp < TC_LOAD_WARPS) {
            // copies of one round, global -> shared memory, 16 bytes each (zero-filled past the end of the list): this lane's
            // piece of rows warp, warp + 16, ... and (threads 0-255) this thread's 16 bytes of the tokens' values of row tid / 4
            auto copy_round = [&](int mr) {
                const int gr = g + mr;                                      // round number over the whole kernel
                if (mr < n_rounds) {
                    // the MMAs that read this ring slot four rounds ago must be through
                    if (gr >= TC_BUFS && !failed) {
                        if (s.fail || !mbar_wait(&s.done[gr % TC_BUFS], ((gr / TC_BUFS) - 1) & 1, p.wait_limit_ns)) failed = true;
                    }
                    const uint32_t ab = smem_u32(s.a[gr % TC_BUFS]) + a_off;
#pragma unroll
                    for (int u = 0; u < TC_U; ++u) {
                        const int r = mr * TC_ROUND_ROWS + warp + u * TC_LOAD_WARPS;
                        const bool ok = r < n_rows && lane_ok;
                        const char *src = ok ? base + (size_t)s.idx[r] * p.row_bytes : p.W;
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ab + u * TC_A_KB_BYTES), "l"(src),
                                     "r"(ok ? 16 : 0) : "memory");
                    }
                    if (tid < TC_ROUND_ROWS * 4) {
                        const int r = mr * TC_ROUND_ROWS + bb_row;
                        const bool ok = r < n_rows;
                        const uint16_t *src = ok ? q.xt + (size_t)s.idx[r] * 32 + bb_mg * 8 : q.xt;
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(s.b[gr % TC_BUFS]) + b_off), "l"(src),
                                     "r"(ok ? 16 : 0) : "memory");
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");           // (an empty group past the last round)
            };
#pragma unroll
            for (int mr = 0; mr < TC_BUFS - 1; ++mr) copy_round(mr);
            for (int mr = 0; mr < n_rounds; ++mr) {
                // this thread's copies of round mr have landed (the two younger groups may be in flight)
                asm volatile("cp.async.wait_group %0;" ::"n"(TC_BUFS - 2) : "memory");
                // -> visible to the tensor core's (async proxy) reads
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&s.full[(g + mr) % TC_BUFS]);
                copy_round(mr + TC_BUFS - 1);
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");              // (only empty groups are left)
        } else if (lane == 0) {
            // the MMA thread: per round, wait for the 16 loader warps, then one MMA per K-block
            for (int mr = 0; mr < n_rounds; ++mr) {
                const int gg = g + mr, buf = gg % TC_BUFS;
                if (failed) break;
                if (s.fail || !mbar_wait(&s.full[buf], (gg / TC_BUFS) & 1, p.wait_limit_ns)) {
                    failed = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int rows_here = min(TC_ROUND_ROWS, n_rows - mr * TC_ROUND_ROWS);
                const int nkb = (rows_here + 15) >> 4;
                // descriptors of K-block 0; K-block kb is kb * bytes further (start address field in 16-byte units).
                // values: MN-major (token slots contiguous), no swizzle: 8-row groups 128 B apart, the two 8-k groups 2 KB apart;
                // weights: MN-major, 128-byte swizzle: 64-output blocks 1 KB apart, rows 0-7 / 8-15 4 KB apart
                const uint64_t x_d0 = tc_smem_desc(smem_u32(s.b[buf]), 2048, 128, 0);
                const uint64_t w_d0 = tc_smem_desc(smem_u32(s.a[buf]), 1024, 4096, 2);
                for (int kb = 0; kb < nkb; ++kb)
                    tc_mma(tmem, x_d0 + (uint64_t)(kb * (TC_B_KB_BYTES >> 4)), w_d0 + (uint64_t)(kb * (TC_A_KB_BYTES >> 4)),
                           (gg > 0 || kb > 0) ? 1u : 0u);
                tc_commit(&s.done[buf]);
            }
        }
        g += n_rounds;
    }
    DIP_TRACE_MAX(p.tr, 3);            // streaming done
    if (failed) s.fail = 1;
    __syncthreads();
    failed = s.fail != 0;
    // ---- the last round's commit covers every MMA of the kernel ----
    if (g > 0 && !failed) {
        if (!mbar_wait(&s.done[(g - 1) % TC_BUFS], ((g - 1) / TC_BUFS) & 1, p.wait_limit_ns)) failed = true;
    }
    if (failed && lane == 0) atomicExch(p.status, 1);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    // ---- the useful accumulator rows 0-31 are tensor-memory lanes 0-31, which the warps 0, 4, 8 and 12 reach (a warp reads
    //      the lane quarter warp % 4): token n's high-half sums in lane n, the low-half sums in lane 16 + n.  64 packed outputs per
    //      warp, over the ring's first buffer ----
    constexpr int ROW = 256 + 4;
    float *sums = reinterpret_cast<float *>(&s.a[0][0]);           // [token][ROW]
    if ((warp & 3) == 0 && warp < 16) {
        const int c0 = warp;                                       // this warp's columns: 16 c0 .. 16 c0 + 63 (c0 = 0, 4, 8, 12)
        float v[64];
        if (g > 0 && !failed) {
            tc_ld64(tmem + 16 * c0, v);
        } else {
#pragma unroll
            for (int i = 0; i < 64; ++i) v[i] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < 64; ++i) v[i] += __shfl_down_sync(0xffffffffu, v[i], 16);       // + the low halves' sums
        if (lane < p.batch) {
#pragma unroll
            for (int i = 0; i < 64; i += 4)
                *reinterpret_cast<float4 *>(sums + lane * ROW + 16 * c0 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // ---- row parts: for a launch behind this one, or to the last part's CTA, which adds them up in part order (see gemv_fused.cu) ----
    const size_t stride = (size_t)q.n_slabs * p.batch * 256;
    float *box = p.mail + (size_t)slab * p.batch * 256;
    if (p.defer) {
        float *to = p.partials + (size_t)part * stride + (size_t)slab * p.batch * 256;
        for (int e = tid; e < p.batch * 64; e += TC_THREADS)
            *reinterpret_cast<float4 *>(to + 4 * e) = *reinterpret_cast<const float4 *>(sums + (e >> 6) * ROW + 4 * (e & 63));
    } else if (part != nparts - 1) {
        for (int e = tid; e < p.batch * 64; e += TC_THREADS)
            mail_put4(box + (size_t)part * stride + 4 * e, *reinterpret_cast<const float4 *>(sums + (e >> 6) * ROW + 4 * (e & 63)));
    } else {
        if (nparts > 1) {
            for (int e = tid; e < p.batch * 64; e += TC_THREADS) {
                float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int b0 = 0; b0 < nparts - 1; b0 += MAIL_N) {
                    float4 a[MAIL_N];
                    mail_take4<MAIL_N>(box + (size_t)b0 * stride + 4 * e, stride, nparts - 1 - b0, a, p.status, q.block_wait_ns);
#pragma unroll
                    for (int b = 0; b < MAIL_N; ++b) { t.x += a[b].x; t.y += a[b].y; t.z += a[b].z; t.w += a[b].w; }
                }
                float4 &mine = *reinterpret_cast<float4 *>(sums + (e >> 6) * ROW + 4 * (e & 63));
                mine = make_float4(t.x + mine.x, t.y + mine.y, t.z + mine.z, t.w + mine.w);
            }
            __syncthreads();
        }
        // ---- epilogue: four outputs per thread ----
        constexpr int QUADS = WHICH == 0 ? 32 : 64;
        for (int e = tid; e < p.batch * QUADS; e += TC_THREADS) {
            const int n = e / QUADS, o = 4 * (e % QUADS), j = slab * 4 * QUADS + o;
            if (j >= p.d_out) continue;                            // (d_out is a multiple of 32)
            // gate/up: every 16 columns are 8 gate outputs followed by their 8 up outputs
            const float *at = sums + n * ROW + (WHICH == 0 ? (o >> 3) * 16 + (o & 7) : o);
            float4 r = *reinterpret_cast<const float4 *>(at);
            if (WHICH == 0) {
                const float4 up = *reinterpret_cast<const float4 *>(at + 8);
                r = make_float4(silu_f32(r.x) * up.x, silu_f32(r.y) * up.y, silu_f32(r.z) * up.z, silu_f32(r.w) * up.w);
                // top 16 bits of the rank keys |h_j| for the select that follows (no cache with several tokens)
                if (p.key_coarse)
                    *reinterpret_cast<uint2 *>(p.key_coarse + (size_t)n * p.d_out + j) =
                        make_uint2(((__float_as_uint(r.x) & 0x7fffffffu) >> 16) | ((__float_as_uint(r.y) & 0x7fffffffu) & 0xffff0000u),
                                   ((__float_as_uint(r.z) & 0x7fffffffu) >> 16) | ((__float_as_uint(r.w) & 0x7fffffffu) & 0xffff0000u));
            }
            *reinterpret_cast<float4 *>(p.out + (size_t)n * p.d_out + j) = r;
        }
    }
    // ---- free the tensor memory (its last use lies before the barrier above) ----
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TC_TMEM_COLS) : "memory");
    DIP_TRACE_MAX(p.tr, 2);
}

}  // namespace

// One CTA per 512-byte segment and row part.  Rows of more segments than half the SMs need no parts (gate/up, whose segments may be
// more than SMs); otherwise the parts, all resident at once, meet in the last part's CTA (5120 / 17920, down: 4.6 us
// after its last row for 16 tokens, 1.8 for 5; a launch of its own for the sums, 8.6 until the next select could start).  That
// CTA takes parts x tokens KB, and its SM's share of L2's rate makes that the longer way where both are many: 16 tokens,
// union of 1024 / 4096, one segment (16 / 64 parts) 15.0 / 32.4 us and 10.6 / 12.0 with a launch behind; 8 tokens, 16 parts 11.4 and 9.9;
// 3 tokens, 32 parts 11.6 and 10.4.  The other way: 5 tokens, 16 parts 10.3 and 9.7, 18 parts of 8 segments 11.1 and 12.0; 16 tokens, 12 parts
// 14.9 and 16.0.
constexpr int TC_APART_PARTS = 16, TC_APART_KB = 96;
dip_status dip_launch_gemv_tc(dip_ctx *ctx, GemvParams &p, int which, int n_kept_max, cudaStream_t stream)
{
    const int n_slabs = (int)((p.row_bytes + TC_SEG - 1) / TC_SEG);
    const int nparts = row_parts(ctx->sm_count / n_slabs, n_kept_max, TC_ROUND_ROWS);   // at least a round of rows per part
    static_assert(TC_N * 256 <= DIP_MAIL_FLOATS, "");        // (parts only with one CTA per SM: the mail boxes suffice)
    p.defer = nparts >= TC_APART_PARTS && nparts * p.batch >= TC_APART_KB;
    p.part_base = 0;
    if (p.defer) {
        if ((size_t)nparts * n_slabs * p.batch * 256 > ctx->partials_floats) return DIP_ERR_WORKSPACE;
        p.key_coarse = nullptr;                              // (nobody in this launch sees h)
    }
    TcParams q;
    q.n_slabs = n_slabs;
    q.nparts = nparts;
    q.xt = ctx->xt;
    q.block_wait_ns = ctx->block_wait_ns;
    const size_t smem = sizeof(TcSmem) + 1024;
    static_assert(sizeof(TcSmem) + 1024 <= 227 * 1024, "fits a CTA's shared memory");
    static dip_per_device_once once[2];
    const int xt_ctas = min((p.mask_words + 1) / 2, 2 * ctx->sm_count);
    DIP_CUDA_TRY(ctx, dip_launch_pdl(xt_build_kernel, dim3(xt_ctas), dim3(1024), 0, stream, p.mask_bits, p.v, p.batch, p.d_in,
                                     p.mask_words, ctx->xt));
    if (which == 0) {
        DIP_CUDA_TRY(ctx, dip_raise_smem_limit(once[0], ctx->device, gemv_tc_kernel<0>, smem));
        DIP_CUDA_TRY(ctx, dip_launch_pdl(gemv_tc_kernel<0>, dim3(n_slabs * nparts), dim3(TC_THREADS), smem, stream, p, q));
    } else {
        DIP_CUDA_TRY(ctx, dip_raise_smem_limit(once[1], ctx->device, gemv_tc_kernel<1>, smem));
        DIP_CUDA_TRY(ctx, dip_launch_pdl(gemv_tc_kernel<1>, dim3(n_slabs * nparts), dim3(TC_THREADS), smem, stream, p, q));
    }
    if (p.defer) return dip_launch_combine_parts(ctx, which, nparts, n_slabs, p.batch, 256, 8, p.batch, p.d_out, p.out, stream);
    return DIP_OK;
}
