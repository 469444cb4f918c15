// Declarations shared by the product kernels (gemv.cu, gemv_fused.cu, gemv_direct_bt.cu, gemv_int4.cu, gemv_tc.cu).
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

constexpr int GV_MAX_ROWS = 2048;                          // kept rows per round (index list in smem)
constexpr int GV_SCAN_THREADS = 256;                       // threads that scan the mask words

struct GemvParams {
    const char *W;             // packed rows
    size_t row_bytes;          // bytes of one packed row
    const uint16_t *scales;    // INT4: binary16 scales [d_in/128][row elements], laid out like a row
    size_t scale_row_elems;    // INT4: elements of one scale row
    const float *v;            // [batch][d_in]
    int d_in;
    const uint32_t *mask_bits; // [batch][mask_words]; rows read = OR over the batch
    int mask_words;
    const int32_t *list;       // one token: the kept columns as a list of n_list (see dip_launch_gemv) instead of mask_bits
    int n_list;
    float *out;                // [batch][d_out]
    int d_out;
    int batch;                 // tokens in this launch (<= BT)
    float *partials;
    float *mail;               // row parts on their way between CTAs of a launch; DIP_MAIL_EMPTY outside one
    unsigned int *tickets;
    int *status;               // device status word (0 = fine)
    unsigned long long wait_limit_ns;   // a wait on a copy's arrival, or on another block, gives up after this long
    unsigned long long *tr;    // timeline slot or nullptr
    const int32_t *loc;        // two-tier: packed row of column i is W + loc[i] * row_bytes (nullptr: row i)
    int defer;                 // 1: leave the row parts in `partials` for combine_parts_kernel
    int part_base;             // first part index of this launch inside `partials`
    // gate/up, single-token launches only: top 16 bits of the rank key of every h_j for the select
    // that follows (nullptr: not wanted); the key is |h_j| * (key_stamp[j] >= 0 ? 1 : key_gamma),
    // or |h_j| without stamps
    uint16_t *key_coarse;
    const int32_t *key_stamp;
    float key_gamma;
};


__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait for the phase with the given parity; false if limit_ns ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, unsigned long long limit_ns)
{
    const uint32_t a = smem_u32(bar);
    unsigned long long t0 = 0;
    for (unsigned i = 0;; ++i) {
        unsigned ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(a), "r"(parity) : "memory");
        if (ok) return true;
        if ((i & 255u) == 255u) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            else if (now - t0 > limit_ns) return false;
        }
    }
}

// Asks for `bytes` at p to be brought into L2 (a hint: nothing to wait for).  p on a 16-byte boundary, bytes a
// multiple of 16, the range inside one allocation.
__device__ __forceinline__ void l2_prefetch(const void *p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Sums that one CTA of a launch hands to another through global memory: the value itself is the message.
// A box holds DIP_MAIL_EMPTY (a NaN pattern that no arithmetic produces) until its sum arrives; who
// takes a sum empties its box again.
// The block that waits is the last part of its segment.  It cannot keep those that it waits for from running: a launch with
// parts has at most one block per SM, and where something else holds SMs, blocks are started in index order, so the earlier
// parts are running or done when it starts.  The order is what the hardware does, not a promise, hence the limit.
__device__ __forceinline__ void mail_put(float *box, float v)
{
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(box), "f"(v) : "memory");
}
// The sums of the first min(n, N) of the boxes box[0], box[stride], ... (the others: zero).  Waits at most
// limit_ns for them, after which it records status 1 and takes what is there.
template <int N>
__device__ __forceinline__ void mail_take(float *box, size_t stride, int n, float (&a)[N], int *status, unsigned long long limit_ns)
{
    unsigned long long t0 = 0;
    for (unsigned i = 0;; ++i) {
        bool all = true;
#pragma unroll
        for (int q = 0; q < N; ++q) {
            a[q] = 0.f;
            if (q < n) asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(a[q]) : "l"(box + (size_t)q * stride) : "memory");
        }
#pragma unroll
        for (int q = 0; q < N; ++q) all = all && __float_as_uint(a[q]) != DIP_MAIL_EMPTY;
        if (all) break;
        if ((i & 63u) == 63u) {
            const unsigned long long now = dip_gtime();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > limit_ns) {
                atomicExch(status, 1);
                break;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < N; ++q)
        if (q < n) mail_put(box + (size_t)q * stride, __uint_as_float(DIP_MAIL_EMPTY));
}

// Up to MAIL_N row parts are one trip of a segment's threads, one per element.  More are shared out, MAIL_N at a time,
// over the T / SLAB groups of the last part's CTA (all T threads call it): the sum of the n boxes boxes[0], boxes[stride], ...
// of element tid % SLAB, the groups' sums in order of the groups.  (Narrow rows have up to one part per SM, and a trip to L2
// for every eight added up: the down product of 704 rows of 256 BF16 outputs took 12.3 us, with both this and row_parts
// 5.8.)  Out of line: in line it cost the launches that carry cache updates, which are bound by fetching instructions
// already, 0.4 us (one step with caches: 3072 / 8192 19.1 us and 18.8 like this, 5120 / 17920 34.4 and 34.1).
// scratch: T floats of shared memory that nobody reads or writes any more.
constexpr int MAIL_N = 8;
template <int SLAB, int T>
__device__ __noinline__ float mail_sum_wide(float *boxes, size_t stride, int n, float *scratch, int *status, unsigned long long limit_ns)
{
    static_assert(T % SLAB == 0, "");
    const int tid = threadIdx.x, el = tid % SLAB;
    float sum = 0.f;
    for (int q0 = tid / SLAB * MAIL_N; q0 < n; q0 += T / SLAB * MAIL_N) {
        float a[MAIL_N];
        mail_take<MAIL_N>(boxes + (size_t)q0 * stride + el, stride, n - q0, a, status, limit_ns);
#pragma unroll
        for (int q = 0; q < MAIL_N; ++q) sum += a[q];
    }
    scratch[tid] = sum;
    __syncthreads();
    sum = 0.f;
#pragma unroll
    for (int g = 0; g < T / SLAB; ++g) sum += scratch[g * SLAB + el];
    return sum;
}
// The same for n <= MAIL_N by one thread for its element.
__device__ __forceinline__ float mail_sum(float *box, size_t stride, int n, int *status, unsigned long long limit_ns)
{
    float a[MAIL_N], sum = 0.f;
    mail_take<MAIL_N>(box, stride, n, a, status, limit_ns);
#pragma unroll
    for (int q = 0; q < MAIL_N; ++q) sum += a[q];
    return sum;
}

// Parts of n rows by CTAs of `warps` warps, at most `most`: with less than a row per warp a part takes no less time, and one
// more sum has to be collected (176 rows of 256 BF16 outputs: 12.6 us with 148 parts, 4.3 with 5).
static inline int row_parts(int most, int n, int warps)
{
    const int by_rows = n / warps;
    const int parts = most < by_rows ? most : by_rows;
    return parts < 1 ? 1 : parts;
}

// mail_put / mail_take for groups of four.
__device__ __forceinline__ void mail_put4(float *box, const float4 &v)
{
    asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(box), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
template <int N>
__device__ __forceinline__ void mail_take4(float *box, size_t stride, int n, float4 (&a)[N], int *status, unsigned long long limit_ns)
{
    unsigned long long t0 = 0;
    for (unsigned i = 0;; ++i) {
        bool all = true;
#pragma unroll
        for (int q = 0; q < N; ++q) {
            a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q < n)
                asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a[q].x), "=f"(a[q].y), "=f"(a[q].z), "=f"(a[q].w)
                             : "l"(box + (size_t)q * stride) : "memory");
        }
#pragma unroll
        for (int q = 0; q < N; ++q)
            all = all && __float_as_uint(a[q].x) != DIP_MAIL_EMPTY && __float_as_uint(a[q].y) != DIP_MAIL_EMPTY &&
                  __float_as_uint(a[q].z) != DIP_MAIL_EMPTY && __float_as_uint(a[q].w) != DIP_MAIL_EMPTY;
        if (all) break;
        if ((i & 63u) == 63u) {
            const unsigned long long now = dip_gtime();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > limit_ns) {
                atomicExch(status, 1);
                break;
            }
        }
    }
    const float e = __uint_as_float(DIP_MAIL_EMPTY);
#pragma unroll
    for (int q = 0; q < N; ++q)
        if (q < n) mail_put4(box + (size_t)q * stride, make_float4(e, e, e, e));
}

// One more at a counter in global memory, after what this thread (and those it has synchronised with) has read.
__device__ __forceinline__ void count_one(unsigned int *counter)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}
// Waits until the counter has reached n; false (and status 1) if limit_ns ran out.
__device__ __forceinline__ bool wait_count(const unsigned int *counter, unsigned int n, int *status, unsigned long long limit_ns)
{
    unsigned long long t0 = 0;
    for (unsigned i = 0;; ++i) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
        if (v >= n) return true;
        if ((i & 63u) == 63u) {
            const unsigned long long now = dip_gtime();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > limit_ns) {
                atomicExch(status, 1);
                return false;
            }
        }
    }
}

__device__ __forceinline__ float silu_f32(float g) { return g / (1.0f + expf(-g)); }

__device__ __forceinline__ float half_bits_to_float(uint16_t h)
{
    return __half2float(__ushort_as_half(h));
}

// The columns in list[0 .. n) as a bit set: words[] is zero on entry (and that is visible), all T threads call it, no
// barrier at the end.  (Every CTA of a product for itself: a few KB out of L2, against a launch of its own in front.)
template <int T>
__device__ __forceinline__ void list_to_words(const int32_t *list, int n, int d, uint32_t *words)
{
    constexpr int U = 4;                       // loads that go out together
    for (int r0 = threadIdx.x; r0 < n; r0 += U * T) {
        int i[U];
#pragma unroll
        for (int u = 0; u < U; ++u) i[u] = r0 + u * T < n ? __ldg(list + r0 + u * T) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i[u] >= 0 && i[u] < d) atomicOr(&words[i[u] >> 5], 1u << (i[u] & 31));
    }
}

namespace {

template <int WT> struct WTraits;
// E = weights in a lane's 16 bytes; C = gate/up interleave chunk of the bundled rows (weights)
template <> struct WTraits<DIP_W_F32>       { static constexpr int E = 4;  static constexpr int C = 4; };
template <> struct WTraits<DIP_W_BF16>      { static constexpr int E = 8;  static constexpr int C = 8; };

template <int WT> __device__ __forceinline__ void decode16(const uint4 &r, float (&w)[WTraits<WT>::E]);
template <> __device__ __forceinline__ void decode16<DIP_W_F32>(const uint4 &r, float (&w)[4])
{
    w[0] = __uint_as_float(r.x); w[1] = __uint_as_float(r.y);
    w[2] = __uint_as_float(r.z); w[3] = __uint_as_float(r.w);
}
// bfloat16 is the upper half of a binary32: widening is a shift or a mask.
template <> __device__ __forceinline__ void decode16<DIP_W_BF16>(const uint4 &r, float (&w)[8])
{
    const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        w[2 * i] = __uint_as_float(u[i] << 16);
        w[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}

}  // namespace

// gemv.cu: sum of the row parts left in ctx->partials ([parts][n_slabs][bt][slab_elems]; gate/up
// elements interleaved in chunks of c) and the epilogue, spread over the device.
dip_status dip_launch_combine_parts(dip_ctx *ctx, int which, int total_parts, int n_slabs, int bt, int slab_elems, int c,
                                    int batch, int d_out, float *out, cudaStream_t stream);

// gemv_direct_bt.cu: F32 / BF16 weights, two tokens: the product over the union of the tokens' rows with
// plain loads and FMAs.
dip_status dip_launch_gemv_direct_bt(dip_ctx *ctx, GemvParams &p, int wtype, int which, int n_kept_max, cudaStream_t stream);

// gemv_tc.cu: BF16 weights, 8 to 16 tokens: the product over the union of the tokens' rows on tcgen05 tensor cores.
dip_status dip_launch_gemv_tc(dip_ctx *ctx, GemvParams &p, int which, int n_kept_max, cudaStream_t stream);

// gemv_int4.cu: the single-token product for INT4-g128 weights.  mode as dip_gemv_rows.mode.
// sel != nullptr (mode 0): the product builds its own mask, as gemv_fused.cu's do (p.mask_bits is not read).
dip_status dip_launch_gemv_int4(dip_ctx *ctx, GemvParams &p, int which, int n_kept_max, int mode, const dip_fused_select *sel,
                                cudaStream_t stream);
bool dip_gemv_int4_selects(const dip_ctx *ctx, const dip_mlp_weights *w, int which);
