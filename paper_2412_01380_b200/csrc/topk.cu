// Masking kernels: magnitude top-k (Sec. 3.1, Eq. 7-8), the cache-aware ranking of Eq. 10, the
// LRU column-cache update of Algorithm 1, index lists / unions from bit masks, and the residual
// + RMS re-normalisation that chains layers.
//
// The step's critical path only needs the mask, so the work is split in two kernels:
//   select_fine_kernel   rank keys -> k-th largest key by a histogram of their top 15 bits -> bit
//                        mask.  One CTA of 1024 threads per row; the keys live in shared memory.
//   cache_update_kernel  hits, misses, LRU victims and the new stamps from (mask, state).  It
//                        does not feed the GEMVs and runs beside them on another stream.
// Everything here is integer work on bit patterns, so results are exact and unique (ties go
// to the lower column index).
#include "select_core.cuh"

namespace {


// ---------------------------------------------------------------------------------------
// select_fine_kernel: the mask of one row by the one-histogram select of select_core.cuh (the
// select that the fused product kernels run), one CTA per row.
//   CA == false: key = bits(|x|)                              (DIP, Eq. 7-8)
//   CA == true : key = bits(|x| * (resident ? 1 : gamma))     (numerator of Eq. 10); the cache
//                state is only read.
//   NORM == true: the row is first formed as x = (xa + xb) / rms(xa + xb) (the layer chaining
//                of a stack) and written to x_out; the summation order is that of
//                residual_rmsnorm_kernel, so both give the same bits.
// select_fine_coarse_kernel: the same mask as select_fine_kernel<CA, false> for one row whose
// producer has already left the top 16 bits of every rank key in coarse[] (the gate/up product
// does, in its epilogue): one SM reads global memory at a fraction of the device's rate, so the
// bytes this CTA has to pull in are its floor: two bytes per column instead of the eight of value +
// stamp.  Needs d % 8 == 0 and d <= 8 * TK_COARSE_ITERS * TK_THREADS.
// Dynamic shared memory: TkFine, then keys[] (d words rounded up to four).
// ---------------------------------------------------------------------------------------
template <bool CA, bool NORM>
__global__ void __launch_bounds__(TK_THREADS, 1)
select_fine_kernel(const float *__restrict__ xa, const float *__restrict__ xb, float *__restrict__ x_out,
                   int d, int k, float gamma, const int32_t *__restrict__ stamp,
                   uint32_t *__restrict__ mask_bits, unsigned long long *tr)
{
    DIP_TRACE_MIN(tr, 0);
    extern __shared__ __align__(16) unsigned char dyn[];
    TkFine &f = *reinterpret_cast<TkFine *>(dyn);
    uint32_t *keys = reinterpret_cast<uint32_t *>(dyn + sizeof(TkFine));
    __shared__ TkShared s;
    __shared__ unsigned int s_maskw[DIP_MAX_D / 32];
    const int tid = threadIdx.x;
    const int row = blockIdx.x;
    const int n_words = (d + 31) >> 5;
    xa += (size_t)row * d;
    if (NORM) {
        xb += (size_t)row * d;
        x_out += (size_t)row * d;
    }
    mask_bits += (size_t)row * n_words;

    fine_zero(f);
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(tr, 1);
    dip_launch_dependents();
    if (NORM && (d & 3) == 0 && d <= 8 * TK_THREADS) {
        __syncthreads();                                              // histogram zeroed
        select_fine_chained<CA>(xa, xb, x_out, nullptr, d, k, gamma, stamp, keys, s, f, s_maskw);
    } else {
        float scale = 1.0f;
        if (NORM)
            scale = block_residual_scale(xa, xb, d, keys, s.wf, &s.scale);   // ends with a barrier
        else
            __syncthreads();
        select_fine<CA, NORM>(xa, NORM ? x_out : nullptr, nullptr, d, k, gamma, stamp, scale, keys, s, f, s_maskw);
    }
    for (int w = tid; w < n_words; w += TK_THREADS) mask_bits[w] = s_maskw[w];
    DIP_TRACE_MAX(tr, 2);
}

template <bool CA>
__global__ void __launch_bounds__(TK_THREADS, 1)
select_fine_coarse_kernel(const float *__restrict__ x, const uint16_t *__restrict__ coarse, int d, int k, float gamma,
                          const int32_t *__restrict__ stamp, uint32_t *__restrict__ mask_bits, unsigned long long *tr)
{
    DIP_TRACE_MIN(tr, 0);
    extern __shared__ __align__(16) unsigned char dyn[];
    TkFine &f = *reinterpret_cast<TkFine *>(dyn);
    uint32_t *keys = reinterpret_cast<uint32_t *>(dyn + sizeof(TkFine));
    __shared__ TkShared s;
    __shared__ unsigned int s_maskw[DIP_MAX_D / 32];
    const int tid = threadIdx.x;
    const int row = blockIdx.x;                                       // (several rows only without a cache)
    x += (size_t)row * d;
    coarse += (size_t)row * d;
    mask_bits += (size_t)row * (d >> 5);

    fine_zero(f);
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(tr, 1);
    dip_launch_dependents();
    __syncthreads();                                                  // histogram zeroed
    select_fine_coarse<CA>(coarse, x, stamp, gamma, d, k, keys, s, f, s_maskw);
    for (int w = tid; w < (d >> 5); w += TK_THREADS) mask_bits[w] = s_maskw[w];
    DIP_TRACE_MAX(tr, 2);
}

// ---------------------------------------------------------------------------------------
// cache_update_kernel: c' = cache_update(c, m) of Algorithm 1 with the LRU policy of Sec. 5.1
// (or LFU when use counters are given), from the mask bits and the state alone.  One CTA: it runs
// beside a product that fills the other SMs, and a chain of exchanges between CTAs would cost
// more than the few thousand columns an SM has to look at.
// A warp owns NB consecutive blocks of 128 columns, a lane four consecutive columns of each (one
// 16-byte load and one 16-byte store), and everything in between stays in registers.  The eviction
// key of a column that may be evicted (resident and outside the mask) is the age of its last use
// (LFU: t + 1 - uses), of any other column 0.
// Bound by the SM's issue rate and its trips through shared memory.  Alone, LRU, after 38 updates:
// 7.9 us at d = 17920 (load 1.5, histogram 2.1 + search 0.7, ties 1.2, stamps 2.1), 4.4 us at 5120;
// one column per lane swept four times through shared memory with 4-byte stores took 14.4 and 6.6 us.
// ---------------------------------------------------------------------------------------
constexpr int CU_SPREAD = 8;                            // copies of the counters of the small digits,
constexpr int CU_SMALL = 256;                           // which nearly all keys have: ages of a few updates

template <int NB, bool LFU>
__global__ void __launch_bounds__(TK_THREADS, 1)
cache_update_kernel(const uint32_t *__restrict__ mask_bits, int d, int32_t *stamp, int32_t *count, int32_t *meta,
                    int capacity, unsigned long long *tr)
{
    __shared__ TkShared s;
    __shared__ __align__(16) unsigned int small[CU_SMALL * CU_SPREAD];
    static_assert(CU_SMALL * CU_SPREAD == 2 * TK_THREADS && RADIX_BINS == 2 * TK_THREADS, "two counters per thread");
    DIP_TRACE_MIN(tr, 0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const auto clear = [&]() {
        s.hist[2 * tid] = s.hist[2 * tid + 1] = 0;
        small[2 * tid] = small[2 * tid + 1] = 0;
    };
    clear();
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(tr, 1);
    dip_launch_dependents();
    const int n_res = meta[0];
    const int t_now = meta[1] + 1;
    const int col0 = warp * (NB * 128) + lane * 4;      // this lane's first column; block i is 128 i further

    // ---- the state and the mask.  kv: LRU: t_now - stamp (the stamp can be had back), LFU: t_now - uses ----
    uint32_t kv[NB][4];
    uint32_t keep = 0u, res = 0u;                       // nibble i: block i's four columns in the mask / resident
    {
        int st[NB][4], cn[LFU ? NB : 1][4];
        uint32_t word[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int c = col0 + 128 * i;
            word[i] = 0u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                st[i][e] = -1;
                if (LFU) cn[i][e] = 0;
            }
            if (c < d) word[i] = mask_bits[c >> 5];
            if (c + 4 <= d) {
                const int4 q = *reinterpret_cast<const int4 *>(stamp + c);
                st[i][0] = q.x; st[i][1] = q.y; st[i][2] = q.z; st[i][3] = q.w;
                if (LFU) {
                    const int4 n = *reinterpret_cast<const int4 *>(count + c);
                    cn[i][0] = n.x; cn[i][1] = n.y; cn[i][2] = n.z; cn[i][3] = n.w;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (c + e < d) {
                        st[i][e] = stamp[c + e];
                        if (LFU) cn[i][e] = count[c + e];
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int c = col0 + 128 * i;
            uint32_t nib = (word[i] >> ((4 * lane) & 31)) & 0xfu;
            if (c + 4 > d) nib = c < d ? nib & ((1u << (d - c)) - 1u) : 0u;     // no column beyond d
            keep |= nib << (4 * i);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (st[i][e] >= 0) res |= 1u << (4 * i + e);
                // (a column is used at most once per update: uses <= t, so the most rarely used column has the
                // largest key)
                kv[i][e] = (uint32_t)(t_now - (LFU ? cn[i][e] : st[i][e]));
            }
            if (LFU && nib) {                           // used once more (resident or not)
#pragma unroll
                for (int e = 0; e < 4; ++e) cn[i][e] += (int)((nib >> e) & 1u);
                if (c + 4 <= d) {
                    *reinterpret_cast<int4 *>(count + c) = make_int4(cn[i][0], cn[i][1], cn[i][2], cn[i][3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (c + e < d) count[c + e] = cn[i][e];
                }
            }
        }
    }
    const uint32_t may_go = res & ~keep, misses = keep & ~res;
    const auto evict_key = [&](int i, int e) { return (may_go >> (4 * i + e)) & 1u ? kv[i][e] & 0x7fffffffu : 0u; };

    const int warp_hits = __reduce_add_sync(0xffffffffu, __popc(keep & res));
    const int warp_misses = __reduce_add_sync(0xffffffffu, __popc(misses));
    if (lane == 0) {
        s.wa[warp] = warp_hits;
        s.wc[warp] = warp_misses;
    }
    __syncthreads();                                    // the histogram is zero, the counts are there
    int total_hits, total_misses, tot;
    (void)warp_array_prefix(s.wa, warp, lane, total_hits);
    const int miss_before = warp_array_prefix(s.wc, warp, lane, total_misses);
    const int free_slots = capacity - n_res;
    const int evictable = n_res - total_hits;
    const int n_evict = min(max(0, total_misses - free_slots), evictable);
    const int room = free_slots + n_evict;

    // ---- victims: the n_evict largest eviction keys (oldest stamps), lower index first among equals:
    //      radix select from the top bit down, up to 11 bits per pass ----
    uint32_t T2 = 0x7fffffffu;   // no key exceeds it: no victim
    int quota2 = 0, n_eq2 = 0;
    if (n_evict > 0) {
        if (n_evict == evictable) {
            T2 = 0u;             // every evictable column (key > 0) goes
        } else {
            int hi = 32 - __clz(t_now), krem = n_evict;
            uint32_t prefix = 0u, prefix_mask = 0u;
            while (hi > 0) {
                const int w = hi < RADIX_BITS ? hi : RADIX_BITS, shift = hi - w;
                const uint32_t digit_mask = (1u << w) - 1u;
#pragma unroll
                for (int i = 0; i < NB; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t ek = evict_key(i, e);
                        if (ek != 0u && (ek & prefix_mask) == prefix) {
                            const uint32_t dg = (ek >> shift) & digit_mask;
                            atomicAdd(dg < CU_SMALL ? &small[dg * CU_SPREAD + (lane & (CU_SPREAD - 1))] : &s.hist[dg], 1u);
                        }
                    }
                __syncthreads();
                if (tid < CU_SMALL) {
                    const uint4 p = *reinterpret_cast<const uint4 *>(small + tid * CU_SPREAD),
                                q = *reinterpret_cast<const uint4 *>(small + tid * CU_SPREAD + 4);
                    // (all other columns have key 0)
                    s.hist[tid] = p.x + p.y + p.z + p.w + q.x + q.y + q.z + q.w + (tid == 0 && prefix == 0u ? (unsigned)d : 0u);
                }
                __syncthreads();
                find_bin(s, krem);
                prefix |= (uint32_t)s.bcast[0] << shift;
                prefix_mask |= digit_mask << shift;
                krem = s.bcast[1];
                n_eq2 = s.bcast[2];        // after the last pass: the number of keys equal to T2
                hi = shift;
                if (hi > 0) {
                    clear();
                    __syncthreads();
                }
            }
            T2 = prefix;
            quota2 = krem;
        }
    }
    // ---- if only the first quota2 ties go: the ties in front of each warp, and inside the one warp in
    //      which the quota runs out, in front of each lane.  Likewise the misses, if some find no room ----
    uint32_t ties = 0u;
    if (quota2 > 0 && T2 != 0u) {
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (((may_go >> (4 * i + e)) & 1u) && (kv[i][e] & 0x7fffffffu) == T2) ties |= 1u << (4 * i + e);
    }
    // first `quota` of the flagged columns (ascending index) of which `before` lie in earlier warps
    const auto first_of = [&](uint32_t flags, int before, int n_warp, int quota) {
        if (before + n_warp <= quota) return flags;
        if (before >= quota) return 0u;
        uint32_t out = 0u;
        int run = before;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const uint32_t nib = (flags >> (4 * i)) & 0xfu;
            int incl = __popc(nib);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += n;
            }
            int rank = run + incl - __popc(nib);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if ((nib >> e) & 1u) {
                    if (rank < quota) out |= 1u << (4 * i + e);
                    ++rank;
                }
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        return out;
    };
    if (quota2 > 0 && quota2 < n_eq2) {                // (uniform over the block)
        const int warp_ties = __reduce_add_sync(0xffffffffu, __popc(ties));
        if (lane == 0) s.wb[warp] = warp_ties;
        __syncthreads();
        ties = first_of(ties, warp_array_prefix(s.wb, warp, lane, tot), warp_ties, quota2);
    }
    // a hit, or a miss that still finds room (ascending index order), is stamped with this update
    const uint32_t use = (keep & res) | (total_misses > room ? first_of(misses, miss_before, warp_misses, room) : misses);

    // ---- the new stamps ----
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int c = col0 + 128 * i;
        uint32_t gone = 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (evict_key(i, e) > T2) gone |= 1u << e;
        gone |= (ties >> (4 * i)) & 0xfu;
        const uint32_t used = (use >> (4 * i)) & 0xfu;
        if (!(gone | used)) continue;
        if (LFU || c + 4 > d) {
            // (LFU: the old stamps are not kept in registers)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (((gone | used) >> e) & 1u) stamp[c + e] = (gone >> e) & 1u ? -1 : t_now;
        } else {
            int v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                v[e] = (gone >> e) & 1u ? -1 : (used >> e) & 1u ? t_now : t_now - (int)kv[i][e];
            *reinterpret_cast<int4 *>(stamp + c) = make_int4(v[0], v[1], v[2], v[3]);
        }
    }
    if (tid == 0) {
        const int inserted = min(total_misses, room);
        meta[0] = n_res - n_evict + inserted;
        meta[1] = t_now;
        meta[2] += total_hits;
        meta[3] += total_misses;
        meta[4] += n_evict;
        meta[5] += total_misses - inserted;
    }
    DIP_TRACE_MAX(tr, 2);
}

// ---------------------------------------------------------------------------------------
// mask_to_idx_kernel: ascending index list of a bit mask, or of the union of `nb` masks
// (batched decode: the set of weight columns a step reads once).  CTA r handles masks
// r*nb .. r*nb+nb-1 and writes to idx_out + r*out_stride; thread t owns mask word t.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(TK_THREADS, 1)
mask_to_idx_kernel(const uint32_t *__restrict__ mask_bits, int nb, int d,
                   int32_t *__restrict__ idx_out, int out_stride, int32_t *__restrict__ count_out)
{
    __shared__ int wsum[TK_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_words = (d + 31) >> 5;
    mask_bits += (size_t)blockIdx.x * nb * n_words;
    uint32_t u = 0;
    if (tid < n_words)
        for (int b = 0; b < nb; ++b) u |= mask_bits[(size_t)b * n_words + tid];
    int c = __popc(u);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int total;
    int before = warp_array_prefix(wsum, warp, lane, total) + incl - c;
    if (idx_out) {
        int32_t *o = idx_out + (size_t)blockIdx.x * out_stride;
        while (u) {
            int bit = __ffs(u) - 1;
            u &= u - 1;
            o[before++] = tid * 32 + bit;
        }
    }
    if (count_out && tid == 0) count_out[blockIdx.x] = total;
}

// ---------------------------------------------------------------------------------------
// residual_rmsnorm_kernel: x_next = (x + y) / rms(x + y), one CTA per row, fixed summation
// order (per-thread strided partial sums, then a shuffle tree).
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(TK_THREADS, 1)
residual_rmsnorm_kernel(const float *x, const float *y, int d, float *x_next)
{
    __shared__ float wf[TK_WARPS];
    __shared__ float s_scale;
    const int tid = threadIdx.x;
    const size_t off = (size_t)blockIdx.x * d;
    dip_grid_dependency_wait();
    dip_launch_dependents();
    const float sc = block_residual_scale(x + off, y + off, d, nullptr, wf, &s_scale);
    for (int e = tid; e < d; e += TK_THREADS) x_next[off + e] = (x[off + e] + y[off + e]) * sc;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------------------
dip_status dip_launch_select(dip_ctx *ctx, const float *xa, const float *xb, float *x_out, int batch, int d, int k,
                             float gamma, const int32_t *stamp, uint32_t *mask_bits, cudaStream_t stream,
                             const uint16_t *coarse)
{
    const size_t smem = sizeof(TkFine) + (size_t)((d + 3) & ~3) * sizeof(uint32_t);
    const dim3 grid(batch), block(TK_THREADS);
    unsigned long long *tr = dip_trace_slot(ctx, d <= 0 ? 0 : (stamp ? 2 : 1));
    cudaError_t e;
    if (coarse) {
        if (xb || (batch != 1 && stamp) || (d & 31)) return DIP_ERR_INVALID_ARG;
        if (stamp)
            e = dip_launch_pdl(select_fine_coarse_kernel<true>, grid, block, smem, stream, xa, coarse, d, k, gamma, stamp,
                               mask_bits, tr);
        else
            e = dip_launch_pdl(select_fine_coarse_kernel<false>, grid, block, smem, stream, xa, coarse, d, k, 1.0f,
                               (const int32_t *)nullptr, mask_bits, tr);
    } else if (xb) {
        if (stamp)
            e = dip_launch_pdl(select_fine_kernel<true, true>, grid, block, smem, stream, xa, xb, x_out, d, k, gamma, stamp, mask_bits, tr);
        else
            e = dip_launch_pdl(select_fine_kernel<false, true>, grid, block, smem, stream, xa, xb, x_out, d, k, 1.0f,
                               (const int32_t *)nullptr, mask_bits, tr);
    } else {
        if (stamp)
            e = dip_launch_pdl(select_fine_kernel<true, false>, grid, block, smem, stream, xa, (const float *)nullptr,
                               (float *)nullptr, d, k, gamma, stamp, mask_bits, tr);
        else
            e = dip_launch_pdl(select_fine_kernel<false, false>, grid, block, smem, stream, xa, (const float *)nullptr,
                               (float *)nullptr, d, k, 1.0f, (const int32_t *)nullptr, mask_bits, tr);
    }
    DIP_CUDA_TRY(ctx, e);
    return DIP_OK;
}

dip_status dip_launch_cache_update(dip_ctx *ctx, const uint32_t *mask_bits, int d, int32_t *stamp, int32_t *count,
                                   int32_t *meta, int capacity, cudaStream_t stream)
{
    unsigned long long *tr = dip_trace_slot(ctx, 3);
    // blocks of 128 columns per warp: the smallest that covers d (a column's state is a register)
    void (*kernel)(const uint32_t *, int, int32_t *, int32_t *, int32_t *, int, unsigned long long *);
    if (d <= 2 * 128 * TK_WARPS) kernel = count ? cache_update_kernel<2, true> : cache_update_kernel<2, false>;
    else if (d <= 5 * 128 * TK_WARPS) kernel = count ? cache_update_kernel<5, true> : cache_update_kernel<5, false>;
    else kernel = count ? cache_update_kernel<8, true> : cache_update_kernel<8, false>;
    static_assert(DIP_MAX_D <= 8 * 128 * TK_WARPS, "");
    DIP_CUDA_TRY(ctx, dip_launch_pdl(kernel, dim3(1), dim3(TK_THREADS), 0, stream, mask_bits, d, stamp, count, meta, capacity, tr));
    return DIP_OK;
}

// Per-device set-up: the mask kernels keep up to DIP_MAX_D keys in dynamic shared memory.
dip_status dip_init_mask_kernels(dip_ctx *ctx)
{
    const int bytes = DIP_MAX_D * (int)sizeof(uint32_t);
    const int fine_bytes = bytes + (int)sizeof(TkFine);
    DIP_CUDA_TRY(ctx, cudaFuncSetAttribute(select_fine_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes));
    DIP_CUDA_TRY(ctx, cudaFuncSetAttribute(select_fine_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes));
    DIP_CUDA_TRY(ctx, cudaFuncSetAttribute(select_fine_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes));
    DIP_CUDA_TRY(ctx, cudaFuncSetAttribute(select_fine_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes));
    DIP_CUDA_TRY(ctx, cudaFuncSetAttribute(select_fine_coarse_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes));
    DIP_CUDA_TRY(ctx, cudaFuncSetAttribute(select_fine_coarse_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes));
    return DIP_OK;
}

// rows x (OR of nb masks) -> ascending index lists (and their lengths)
dip_status dip_launch_mask_to_idx(dip_ctx *ctx, const uint32_t *mask_bits, int rows, int nb, int d,
                                  int32_t *idx_out, int out_stride, int32_t *count_out, cudaStream_t stream)
{
    mask_to_idx_kernel<<<rows, TK_THREADS, 0, stream>>>(mask_bits, nb, d, idx_out, out_stride, count_out);
    DIP_CUDA_TRY(ctx, cudaGetLastError());
    return DIP_OK;
}

dip_status dip_launch_residual_rmsnorm(dip_ctx *ctx, const float *x, const float *y, int batch, int d,
                                       float *x_next, cudaStream_t stream)
{
    DIP_CUDA_TRY(ctx, dip_launch_pdl(residual_rmsnorm_kernel, dim3(batch), dim3(TK_THREADS), 0, stream, x, y, d, x_next));
    return DIP_OK;
}
