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
#include <type_traits>

#include "cache_update.cuh"

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
// LIST: the kept columns of row r as an ascending list at idx_out + r * k, LIST_SHORT straight from the mask, LIST_LONG through shared memory
// (variants, since code beside it costs a launch that does not use it 0.1 to 0.25 us).
// THEN (one row): THEN_UPDATE: the CTA goes on to update the row's cache (Algorithm 1 whole).  What bounds dip_ca_mask is the chain of
// its launches (select, update and list were three), and the mask is here in shared memory: masks with lists and list
// products at 2080 / 5472, four calls in a graph, 36.7 us with ten launches and 28.8 with four.  (In line the update spills 308 bytes; as a
// function of its own it spills none and takes longer: 1280 of 5120 columns 6.3 us in line and 6.8, 4480 of 17920 11.3 and 12.3.)
// THEN_SPLIT: it goes on to part the mask into the tier's hits (columns in a slot, whose arena rows go to loc) and its misses (a
// list; their arena rows are the staging rows, in order).
// ---------------------------------------------------------------------------------------
constexpr int THEN_NOTHING = 0, THEN_UPDATE = 1, THEN_SPLIT = 2;
constexpr int LIST_NONE = 0, LIST_SHORT = 1, LIST_LONG = 2;
struct ThenSplit {
    dip_tier t;
    unsigned int *moves;       // the word in which the launch behind says that its moves are known: 0 from here on
};
template <int THEN> using ThenArg = std::conditional_t<THEN == THEN_UPDATE, dip_cache_update, std::conditional_t<THEN == THEN_SPLIT, ThenSplit, Int<0>>>;

template <bool CA, bool NORM, int THEN, int LIST>
__global__ void __launch_bounds__(TK_THREADS, 1)
select_fine_kernel(const float *__restrict__ xa, const float *__restrict__ xb, float *__restrict__ x_out,
                   int d, int k, float gamma, const int32_t *stamp,
                   uint32_t *__restrict__ mask_bits, int32_t *__restrict__ idx_out,
                   const ThenArg<THEN> then, unsigned long long *tr)
{
    static_assert(THEN == THEN_NOTHING || (CA && !NORM), "");
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
        select_fine_chained<CA>(xa, xb, x_out, d, k, gamma, stamp, keys, s, f, s_maskw);
    } else {
        float scale = 1.0f;
        if (NORM)
            scale = block_residual_scale(xa, xb, d, keys, s.wf, &s.scale);   // ends with a barrier
        else
            __syncthreads();
        select_fine<CA, NORM>(xa, NORM ? x_out : nullptr, d, k, gamma, stamp, scale, keys, s, f, s_maskw);
    }
    for (int w = tid; w < n_words; w += TK_THREADS) mask_bits[w] = s_maskw[w];
    if constexpr (LIST != LIST_NONE) {
        static_assert(sizeof(f.hist) >= sizeof(uint16_t) * DIP_MAX_D, "the list fits where the histogram was");
        write_list<LIST == LIST_LONG>(s_maskw, d, k, s, reinterpret_cast<uint16_t *>(f.hist), idx_out + (size_t)row * k);
    }
    if constexpr (THEN == THEN_UPDATE) {
        cache_update_clear(s, f.hist);
        block_cache_update_any(s_maskw, d, then.stamp, then.stamp, then.count, then.meta, then.capacity, s, f.hist, []() {},
                               []() { return true; });
    }
    if constexpr (THEN == THEN_SPLIT) {
        const dip_tier &tier = then.t;
        // a mask word per warp, a column per lane (d is a multiple of 32 here)
        const int lane = tid & 31, warp = tid >> 5;
        unsigned int *missw = f.hist;
        constexpr int U = 8;                       // words whose loads go out together
        for (int w0 = warp; w0 < n_words; w0 += U * TK_WARPS) {
            int sl[U];
#pragma unroll
            for (int v = 0; v < U; ++v) sl[v] = w0 + v * TK_WARPS < n_words ? tier.slot[(w0 + v * TK_WARPS) * 32 + lane] : -1;
#pragma unroll
            for (int v = 0; v < U; ++v) {
                const int w = w0 + v * TK_WARPS;
                if (w >= n_words) break;
                const uint32_t m = s_maskw[w];
                const bool hit = ((m >> lane) & 1u) && sl[v] >= 0 && sl[v] < tier.capacity;   // (a slot outside the arena is none)
                const uint32_t hits = __ballot_sync(0xffffffffu, hit);
                if (hit) tier.loc[w * 32 + lane] = sl[v];
                if (lane == 0) {
                    tier.split[w] = hits;
                    tier.split[n_words + w] = missw[w] = m & ~hits;
                }
            }
        }
        __syncthreads();
        const int n = list_mask(missw, d, s, [&](int r, int col) {
            tier.fetch[4 + r] = col;
            tier.loc[col] = tier.capacity + r;
        });
        if (tid == 0) {
            tier.fetch[0] = n;
            *then.moves = 0u;
        }
    }
    DIP_TRACE_MAX(tr, 2);
}

template <bool CA, int LIST>
__global__ void __launch_bounds__(TK_THREADS, 1)
select_fine_coarse_kernel(const float *__restrict__ x, const uint16_t *__restrict__ coarse, int d, int k, float gamma,
                          const int32_t *__restrict__ stamp, uint32_t *__restrict__ mask_bits, int32_t *__restrict__ idx_out,
                          unsigned long long *tr)
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
    if constexpr (LIST != LIST_NONE) write_list<LIST == LIST_LONG>(s_maskw, d, k, s, reinterpret_cast<uint16_t *>(f.hist), idx_out + (size_t)row * k);
    DIP_TRACE_MAX(tr, 2);
}

// ---------------------------------------------------------------------------------------
// cache_update_kernel: block_cache_update (cache_update.cuh) as a launch of its own, a block per cache.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(TK_THREADS, 1)
cache_update_kernel(const dip_cache_updates u, unsigned long long *tr)
{
    __shared__ TkShared s;
    __shared__ __align__(16) unsigned int small[CU_SMALL * CU_SPREAD];
    DIP_TRACE_MIN(tr, 0);
    cache_update_clear(s, small);
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(tr, 1);
    dip_launch_dependents();
    const dip_cache_update &c = u.at[blockIdx.x];
    block_cache_update_any(c.mask, c.d, c.stamp, c.stamp, c.count, c.meta, c.capacity, s, small, []() {}, []() { return true; });
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
    dip_grid_dependency_wait();
    dip_launch_dependents();
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
                             const uint16_t *coarse, int32_t *idx_out, const dip_cache_update *update, const dip_tier *split)
{
    if ((update || split) && (coarse || xb)) return DIP_ERR_INVALID_ARG;
    if (idx_out && xb) return DIP_ERR_INVALID_ARG;
    if ((update || split) && (batch != 1 || !stamp)) return DIP_ERR_INVALID_ARG;
    const int list = !idx_out ? LIST_NONE : k <= TK_LIST_DIRECT ? LIST_SHORT : LIST_LONG;
    const Int<0> no;
    const size_t smem = sizeof(TkFine) + (size_t)((d + 3) & ~3) * sizeof(uint32_t);
    const dim3 grid(batch), block(TK_THREADS);
    unsigned long long *tr = dip_trace_slot(ctx, d <= 0 ? 0 : (stamp ? 2 : 1));
    cudaError_t e;
    if (!stamp) gamma = 1.0f;
    // (a variant per kind of list)
    const auto fine = [&](auto *none, auto *direct, auto *staged, const auto &then) {
        return dip_launch_pdl(list == LIST_NONE ? none : list == LIST_SHORT ? direct : staged, grid, block, smem, stream, xa, xb, x_out, d, k,
                              gamma, stamp, mask_bits, idx_out, then, tr);
    };
    const auto fine_coarse = [&](auto *none, auto *direct, auto *staged) {
        return dip_launch_pdl(list == LIST_NONE ? none : list == LIST_SHORT ? direct : staged, grid, block, smem, stream, xa, coarse, d, k,
                              gamma, stamp, mask_bits, idx_out, tr);
    };
    if (coarse) {
        if (xb || (batch != 1 && stamp) || (d & 31)) return DIP_ERR_INVALID_ARG;
        e = stamp ? fine_coarse(select_fine_coarse_kernel<true, 0>, select_fine_coarse_kernel<true, 1>, select_fine_coarse_kernel<true, 2>)
                  : fine_coarse(select_fine_coarse_kernel<false, 0>, select_fine_coarse_kernel<false, 1>, select_fine_coarse_kernel<false, 2>);
    } else if (xb) {
        const auto one = [&](auto *kernel) { return fine(kernel, kernel, kernel, no); };
        e = stamp ? one(select_fine_kernel<true, true, THEN_NOTHING, 0>) : one(select_fine_kernel<false, true, THEN_NOTHING, 0>);
    } else if (update) {
        e = fine(select_fine_kernel<true, false, THEN_UPDATE, 0>, select_fine_kernel<true, false, THEN_UPDATE, 1>,
                 select_fine_kernel<true, false, THEN_UPDATE, 2>, *update);
    } else if (split) {
        if (idx_out) return DIP_ERR_INVALID_ARG;
        const auto one = [&](auto *kernel) { return fine(kernel, kernel, kernel, ThenSplit{*split, ctx->readers + 1}); };
        e = one(select_fine_kernel<true, false, THEN_SPLIT, 0>);
    } else if (stamp) {
        e = fine(select_fine_kernel<true, false, THEN_NOTHING, 0>, select_fine_kernel<true, false, THEN_NOTHING, 1>,
                 select_fine_kernel<true, false, THEN_NOTHING, 2>, no);
    } else {
        e = fine(select_fine_kernel<false, false, THEN_NOTHING, 0>, select_fine_kernel<false, false, THEN_NOTHING, 1>,
                 select_fine_kernel<false, false, THEN_NOTHING, 2>, no);
    }
    DIP_CUDA_TRY(ctx, e);
    return DIP_OK;
}

dip_status dip_launch_cache_updates(dip_ctx *ctx, const dip_cache_updates &u, cudaStream_t stream)
{
    if (u.n < 1) return DIP_OK;
    DIP_CUDA_TRY(ctx, dip_launch_pdl(cache_update_kernel, dim3(u.n), dim3(TK_THREADS), 0, stream, u, dip_trace_slot(ctx, 3)));
    return DIP_OK;
}

// Per-device set-up: the mask kernels keep up to DIP_MAX_D keys in dynamic shared memory.
dip_status dip_init_mask_kernels(dip_ctx *ctx)
{
    const int bytes = DIP_MAX_D * (int)sizeof(uint32_t);
    const int fine_bytes = bytes + (int)sizeof(TkFine);
    cudaError_t e = cudaSuccess;
    const auto raise = [&](auto *...kernels) {
        ((e = e == cudaSuccess ? cudaFuncSetAttribute(kernels, cudaFuncAttributeMaxDynamicSharedMemorySize, fine_bytes) : e), ...);
    };
    raise(select_fine_kernel<true, false, THEN_UPDATE, 0>, select_fine_kernel<true, false, THEN_UPDATE, 1>, select_fine_kernel<true, false, THEN_UPDATE, 2>,
          select_fine_kernel<true, false, THEN_SPLIT, 0>, select_fine_kernel<true, true, THEN_NOTHING, 0>, select_fine_kernel<false, true, THEN_NOTHING, 0>,
          select_fine_kernel<true, false, THEN_NOTHING, 0>, select_fine_kernel<true, false, THEN_NOTHING, 1>, select_fine_kernel<true, false, THEN_NOTHING, 2>,
          select_fine_kernel<false, false, THEN_NOTHING, 0>, select_fine_kernel<false, false, THEN_NOTHING, 1>, select_fine_kernel<false, false, THEN_NOTHING, 2>,
          select_fine_coarse_kernel<true, 0>, select_fine_coarse_kernel<true, 1>, select_fine_coarse_kernel<true, 2>,
          select_fine_coarse_kernel<false, 0>, select_fine_coarse_kernel<false, 1>, select_fine_coarse_kernel<false, 2>);
    DIP_CUDA_TRY(ctx, e);
    return DIP_OK;
}

// rows x (OR of nb masks) -> ascending index lists (and their lengths)
dip_status dip_launch_mask_to_idx(dip_ctx *ctx, const uint32_t *mask_bits, int rows, int nb, int d,
                                  int32_t *idx_out, int out_stride, int32_t *count_out, cudaStream_t stream)
{
    DIP_CUDA_TRY(ctx, dip_launch_pdl(mask_to_idx_kernel, dim3(rows), dim3(TK_THREADS), 0, stream, mask_bits, nb, d, idx_out, out_stride,
                                     count_out));
    return DIP_OK;
}

dip_status dip_launch_residual_rmsnorm(dip_ctx *ctx, const float *x, const float *y, int batch, int d,
                                       float *x_next, cudaStream_t stream)
{
    DIP_CUDA_TRY(ctx, dip_launch_pdl(residual_rmsnorm_kernel, dim3(batch), dim3(TK_THREADS), 0, stream, x, y, d, x_next));
    return DIP_OK;
}
