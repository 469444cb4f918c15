// Two-tier execution (Sec. 5: cached columns in a small fast memory, the rest read from a large
// slow one on a miss).  The cache state says which columns are resident; the kernels here keep
// the table of where they are (slots of an arena in device memory) and bring the missing ones in.
//
// Per masked input the select's CTA parts its mask into hits and misses (topk.cu), and one launch does the rest: block 0 keeps the
// books (Algorithm 1's update, then slots for the columns that became resident), the others are the product.  A few
// warps of each read the misses straight from the slow tier, multiply them and leave their piece of every such row in the staging
// row, while the other warps take the hits out of the arena; when block 0 has said which of the staged rows the cache
// keeps, each block moves its pieces of them.  What bounds a step is the slow tier's rate and a chain of launches: with launches
// for split, list, fetch, update, slots, moves, hits, misses and sums on three streams, a step of 3072 / 8192 (BF16, keep ratio
// 0.25, budget 0.5, tokens correlated by 0.95) took 72 us, of which the host needed all and the device 43; two launches
// per input take 31 (host 20.5, device 28.5).
// Products that cannot read the slow tier themselves (4-bit weights, whose kernel has no room for a block of 1024 threads
// beside it; the copy ring) run beside tier_fetch_kernel and once more over the misses.
#include "cache_update.cuh"
#include "gemv_common.cuh"

namespace {

constexpr int TA_WORDS = DIP_MAX_D / 32;

struct TierParams {
    int d, capacity, staging;
    unsigned long long row_bytes;
    const uint32_t *mask;      // [words] the step's mask
    const uint32_t *split;     // [2][words] its hits, its misses
    int32_t *slot;             // [d] in: slots before the update; out: after it
    int32_t *fetch;            // [0] = misses, [1] = out: rows that move into slots, [4 ..) the misses' columns,
                               // [4 + staging ..) out: the slot that the row of each miss moves to, or -1
    const int32_t *loc;        // [d] arena row of each kept column
    const char *backing;
    char *arena;
    unsigned long long *counters;
    dip_cache_update cache;
    unsigned int *moves;       // 1 once fetch[1] and the moves are there; the select in front of the launch has made it 0
    int *status;
    unsigned long long wait_limit_ns;
    unsigned long long *tr_book, *tr_fetch;
};

struct __align__(16) BookSmem {
    TkShared ts;
    __align__(16) unsigned int small[CU_SMALL * CU_SPREAD];   // (read 16 bytes at a time)
    uint32_t before[TA_WORDS], after[TA_WORDS], free_[TA_WORDS];
    int free_pre[TA_WORDS];
    int ws[3][TK_WARPS];
    int bad;
};

// One block, after the cache update.  Compares the slot table (residency before the update) with the stamps (residency
// after it): evicted columns give up their slots, inserted columns take the lowest free slots in ascending column order.
// Only slots that no column of the mask has become free (its hits are pinned), so the moves may run beside the hits' product.
__device__ __forceinline__ void assign_slots(const TierParams &t, BookSmem &s)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int words = (t.d + 31) / 32;
    const int32_t *stamp = t.cache.stamp;
    s.free_[tid] = 0u;                             // (first the slots that stay taken)
    if (tid == 0) s.bad = 0;
    __syncthreads();                               // the stamps are written, too

    constexpr int U = 8;                           // iterations whose loads are issued together
    for (int base0 = warp * 32; base0 < t.d; base0 += TK_THREADS * U) {
        int slv[U], stv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = base0 + u * TK_THREADS + lane;
            slv[u] = i < t.d ? t.slot[i] : -1;
            stv[u] = i < t.d ? stamp[i] : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int base = base0 + u * TK_THREADS, i = base + lane;
            if (base >= t.d) break;                            // uniform over the warp
            const int sl = slv[u];
            const bool before = sl >= 0, after = stv[u] >= 0;
            const uint32_t bw = __ballot_sync(0xffffffffu, before), aw = __ballot_sync(0xffffffffu, after);
            if (lane == 0) {
                s.before[base >> 5] = bw;
                s.after[base >> 5] = aw;
            }
            if (before && after) {
                if (sl < t.capacity) atomicOr(&s.free_[sl >> 5], 1u << (sl & 31));
                else s.bad = 1;                                // a slot outside the arena
            }
            if (before && !after) t.slot[i] = -1;              // evicted
        }
    }
    __syncthreads();

    const int w = tid;
    uint32_t m = 0u, B = 0u, A = 0u, fr = 0u;
    if (w < words) {
        m = t.mask[w];
        B = s.before[w];
        A = s.after[w];
    }
    if (w * 32 < t.capacity) {
        fr = ~s.free_[w];
        if (t.capacity - w * 32 < 32) fr &= (1u << (t.capacity - w * 32)) - 1u;
    }
    const uint32_t ins = ~B & A;           // became resident in this step
    const uint32_t miss = m & ~B;          // kept and not resident before: fetched into staging
    if ((ins & ~miss) | (m & B & ~A)) s.bad = 1;   // only misses are inserted; the mask's hits stay
    const int v[3] = {__popc(ins), __popc(miss), __popc(fr)};
    int pre[3], tot[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        pre[c] = v[c];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, pre[c], o);
            if (lane >= o) pre[c] += n;
        }
        if (lane == 31) s.ws[c][warp] = pre[c];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const unsigned x = (unsigned)s.ws[c][lane];
        pre[c] += (int)__reduce_add_sync(0xffffffffu, lane < warp ? x : 0u) - v[c];
        tot[c] = (int)__reduce_add_sync(0xffffffffu, x);
    }
    s.free_[w] = fr;
    s.free_pre[w] = pre[2];
    const bool bad = s.bad || tot[0] > tot[2] || tot[1] > t.staging;
    __syncthreads();
    int32_t *move = t.fetch + 4 + t.staging;
    if (bad) {
        // the table and the cache state disagree: move nothing, say so
        for (int r = tid; r < t.staging; r += TK_THREADS) move[r] = -1;
        if (tid == 0) {
            t.fetch[1] = 0;
            atomicExch(t.status, 2);
        }
        return;
    }
    int r = pre[1], j = pre[0];                    // rank among the misses = staging row; rank among the inserted columns
    for (uint32_t u = miss; u; u &= u - 1, ++r) {
        const int bit = __ffs(u) - 1;
        int sl = -1;
        if ((ins >> bit) & 1u) {
            // the j-th inserted column takes the j-th free slot: the last word with at most j free ones in front of it
            int a = 0;
#pragma unroll
            for (int step = TA_WORDS / 2; step > 0; step >>= 1)
                if (s.free_pre[a + step] <= j) a += step;
            uint32_t f = s.free_[a];
            for (int q = j - s.free_pre[a]; q > 0; --q) f &= f - 1;
            sl = a * 32 + __ffs(f) - 1;
            t.slot[w * 32 + bit] = sl;
            ++j;
        }
        move[r] = sl;
    }
    if (tid == 0) {
        t.fetch[1] = tot[0];
        t.counters[0] += (unsigned long long)tot[1];
        t.counters[1] += (unsigned long long)tot[1] * t.row_bytes;
    }
}

// Block 0 of a launch: update, slots, moves.  In line, though its registers do not fit beside the product's (364 to 392 bytes of spills): as a
// function of its own that spills nothing it is slower to call than the spills are (one step, keep ratio 0.25, budget 0.5: BF16 3072 / 8192
// 30.9 us in line and 32.6, 5120 / 17920 52.2 and 54.6).
__device__ __forceinline__ void keep_books(const TierParams &t, BookSmem &s)
{
    const dip_cache_update &c = t.cache;
    DIP_TRACE_MIN(t.tr_book, 0);
    cache_update_clear(s.ts, s.small);
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(t.tr_book, 1);
    dip_launch_dependents();
    block_cache_update_any(c.mask, c.d, c.stamp, c.stamp, c.count, c.meta, c.capacity, s.ts, s.small, []() {}, []() { return true; });
    assign_slots(t, s);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        count_one(t.moves);
    }
    DIP_TRACE_MAX(t.tr_book, 2);
}

// The blocks that move rows wait here for block 0, which has started before them (blocks start in index order).  False (and
// status 1) if that takes longer than the limit: then the slot table may name rows that have not moved.
__device__ __forceinline__ bool moves_known(const TierParams &t, int *go)
{
    if (threadIdx.x == 0) *go = wait_count(t.moves, 1u, t.status, t.wait_limit_ns);
    __syncthreads();
    return *go != 0;
}

// ---------------------------------------------------------------------------------------------
// tier_fetch_kernel: block 0 keeps the books, the other warps copy the missing rows from the slow tier into the staging rows and, of
// those that the cache keeps, into their slots, 2 KB a time (16 bytes per lane, four loads in flight; plain loads, since the source may be host
// memory mapped into the device's address space).  A megabyte in flight covers the host link many times over, and
// the other SMs are the product's.  The product of the misses waits for this launch, so nothing may stand behind its last read: a warp
// waits for block 0 while its first piece is under way (10 us, the reads take 30) and has both places of each piece then.  With a second
// pass that moved staged rows to their slots a step of 4096 / 14336 with 4-bit weights took 99.2 us, 92.5 like this (nine launches: 96.9).
// ---------------------------------------------------------------------------------------------
constexpr int TF_PIECE = 2048;

__global__ void __launch_bounds__(TK_THREADS, 1)
tier_fetch_kernel(const TierParams t)
{
    __shared__ BookSmem s;
    if (blockIdx.x == 0) {
        keep_books(t, s);
        return;
    }
    DIP_TRACE_MIN(t.tr_fetch, 0);
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(t.tr_fetch, 1);
    dip_launch_dependents();
    const int lane = threadIdx.x & 31, warp = (int)(blockIdx.x - 1) * TK_WARPS + (threadIdx.x >> 5), n_warps = (int)(gridDim.x - 1) * TK_WARPS;
    const int32_t *cols = t.fetch + 4, *move = t.fetch + 4 + t.staging;
    const int n = min(t.fetch[0], t.staging);
    const int per_row = (int)((t.row_bytes + TF_PIECE - 1) / TF_PIECE);
    const auto load = [&](const char *src, int piece, uint4 (&q)[TF_PIECE / 512]) {
#pragma unroll
        for (int j = 0; j < TF_PIECE / 512; ++j) {
            const size_t at = (size_t)piece * TF_PIECE + j * 512 + lane * 16;
            if (at < t.row_bytes) q[j] = __ldcs(reinterpret_cast<const uint4 *>(src + at));
        }
    };
    const auto store = [&](int row, int piece, const uint4 (&q)[TF_PIECE / 512]) {
        char *dst = t.arena + (size_t)row * t.row_bytes;
#pragma unroll
        for (int j = 0; j < TF_PIECE / 512; ++j) {
            const size_t at = (size_t)piece * TF_PIECE + j * 512 + lane * 16;
            if (at < t.row_bytes) *reinterpret_cast<uint4 *>(dst + at) = q[j];
        }
    };
    bool asked = false, known = false;
    for (long long u = warp; u < (long long)n * per_row; u += n_warps) {
        const int e = (int)(u / per_row), piece = (int)(u % per_row);
        uint4 q[TF_PIECE / 512];
        load(t.backing + (size_t)cols[e] * t.row_bytes, piece, q);
        if (!asked) {                  // (if that takes longer than the limit, the slot table may name rows that are not there)
            asked = true;
            int go = 0;
            if (lane == 0) go = wait_count(t.moves, 1u, t.status, t.wait_limit_ns);
            known = __shfl_sync(0xffffffffu, go, 0) != 0;
        }
        const int sl = known ? __ldcg(move + e) : -1;
        store(t.capacity + e, piece, q);
        if (sl >= 0) store(sl, piece, q);
    }
    DIP_TRACE_MAX_WARP(t.tr_fetch, 2);
}

// ---------------------------------------------------------------------------------------------
// tier_product_kernel: block 0 keeps the books; block 1 + part * n_slabs + slab owns segment `slab` of the packed rows and a
// share of the hits and of the misses.  It streams as gemv_direct_kernel does, and its sums meet the same way.
// Up to TP_MISS_WARPS warps take misses only: the slow tier needs few loads in flight (50 GB/s times some microseconds), and a warp that
// waits for it should not hold up hits.  With no hits all warps take misses.
// ---------------------------------------------------------------------------------------------
constexpr int TP_SEG = 512;
constexpr int TP_U = 4;                            // rows in flight per lane
constexpr int TP_ROWS = 2048;                      // hits and misses per round
constexpr int TP_MISS_WARPS = 8;

struct TierProduct {
    int d_out, n_slabs, nparts;
    const float *v;
    float *out;
    float *mail;
    unsigned long long *tr;
};

struct __align__(16) ProductSmem {
    uint32_t words[2][TA_WORDS];                   // hits, misses
    int pre[2][TA_WORDS];
    int wsum[2][TK_WARPS];
    int total[2];
    uint16_t col[2][TP_ROWS];                      // the round's columns
    uint16_t row[TP_ROWS];                         // the hits' arena rows (< 2 * DIP_MAX_D = 2^16)
    float red[TK_WARPS][32 * 8];                   // [warp][lane * E + e], E <= 8
    float sum[32 * 8];
    int go;
};

// Hits and misses share a block's warps, so fewer of them take the hits and their chains are longer than in a product of hits
// alone.  What that costs in roundings is saved where the sums meet: N sums pairs first, log2(N) roundings instead of N - 1, and the row
// parts with their rounding errors carried along.  Against 64 bits, mean of 24 steps, gate/up and down, in 1e-9:
// BF16 1024 / 2816, keep ratio 0.25: 190 and 127 with sums one after the other, 115 and 75 like this (126 and 99 as two products);
// F32 3072 / 8192, 0.5: 269 and 157, 220 and 116 (299 and 150).
template <int N>
__device__ __forceinline__ float tree_sum(const float *at, int stride)
{
    if constexpr (N == 1) return *at;
    else return tree_sum<N / 2>(at, stride) + tree_sum<N / 2>(at + N / 2 * stride, stride);
}

struct ExactSum {
    float s, c = 0.f;              // the sum in binary32 and the sum of its rounding errors (Knuth's two-sum)
    __device__ __forceinline__ explicit ExactSum(float first) : s(first) {}
    __device__ __forceinline__ void add(float a)
    {
        const float t = __fadd_rn(s, a), b = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(a, b)));
        s = t;
    }
    __device__ __forceinline__ float value() const { return isfinite(s) ? s + c : s; }
};

// own + boxes[0] + boxes[stride] + ... (n > MAIL_N of them) of element tid % SLAB, for threads tid < SLAB; as mail_sum_wide.
template <int SLAB>
__device__ __noinline__ float many_parts(float *boxes, size_t stride, int n, float own, float *scratch, int *status, unsigned long long limit_ns)
{
    const int tid = threadIdx.x, el = tid % SLAB;
    ExactSum mine(0.f);
    for (int q0 = tid / SLAB * MAIL_N; q0 < n; q0 += TK_THREADS / SLAB * MAIL_N) {
        float a[MAIL_N];
        mail_take<MAIL_N>(boxes + (size_t)q0 * stride + el, stride, n - q0, a, status, limit_ns);
#pragma unroll
        for (int q = 0; q < MAIL_N; ++q) mine.add(a[q]);
    }
    scratch[tid] = mine.value();
    __syncthreads();
    ExactSum all(own);
#pragma unroll
    for (int g = 0; g < TK_THREADS / SLAB; ++g) all.add(scratch[g * SLAB + el]);
    return all.value();
}

template <int WT, int WHICH>
__global__ void __launch_bounds__(TK_THREADS, 1)
tier_product_kernel(const TierParams t, const TierProduct p)
{
    constexpr int E = WTraits<WT>::E, C = WTraits<WT>::C;
    constexpr int SLAB = 32 * E;                              // packed elements per segment
    constexpr int OUT_PER_SLAB = WHICH == 0 ? SLAB / 2 : SLAB;
    extern __shared__ __align__(16) unsigned char dyn[];
    if (blockIdx.x == 0) {
        keep_books(t, *reinterpret_cast<BookSmem *>(dyn));
        return;
    }
    ProductSmem &s = *reinterpret_cast<ProductSmem *>(dyn);
    DIP_TRACE_MIN(p.tr, 0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slab = (int)(blockIdx.x - 1) % p.n_slabs, part = (int)(blockIdx.x - 1) / p.n_slabs, nparts = p.nparts;
    const size_t byte_off = (size_t)slab * TP_SEG + lane * 16;
    const bool lane_ok = byte_off < t.row_bytes;
    const int words = t.d >> 5;
    dip_grid_dependency_wait();
    DIP_TRACE_MIN(p.tr, 1);
    dip_launch_dependents();

    // ---- 1. the words of the hits and of the misses, a thread each, and their popcount prefixes ----
    {
        uint32_t u[2] = {0u, 0u};
        int c[2], incl[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (tid < words) s.words[q][tid] = u[q] = t.split[q * words + tid];
            c[q] = incl[q] = __popc(u[q]);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, incl[q], o);
                if (lane >= o) incl[q] += n;
            }
            if (lane == 31) s.wsum[q][warp] = incl[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const unsigned x = (unsigned)s.wsum[q][lane];
            const int before = (int)__reduce_add_sync(0xffffffffu, lane < warp ? x : 0u);
            s.pre[q][tid] = before + incl[q] - c[q];
            if (tid == TK_THREADS - 1) s.total[q] = before + incl[q];
        }
    }
    __syncthreads();
    int lo[2], hi[2];                              // this part's ranks
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        lo[q] = (int)((long long)part * s.total[q] / nparts);
        hi[q] = (int)((long long)(part + 1) * s.total[q] / nparts);
    }

    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    for (int r0 = 0; r0 < max(hi[0] - lo[0], hi[1] - lo[1]); r0 += TP_ROWS) {
        int n[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) n[q] = max(0, min(hi[q] - lo[q] - r0, TP_ROWS));
        if (r0) __syncthreads();
        // ---- 2. the round's rows in rank order: a thread has a byte of a word ----
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int first = lo[q] + r0, last = first + n[q];
            for (int b = tid; b < 4 * words; b += TK_THREADS) {
                const int w = b >> 2, low = 8 * (b & 3);
                const uint32_t all = s.words[q][w];
                uint32_t u = all & (0xffu << low);
                int rank = s.pre[q][w] + __popc(all & ((1u << low) - 1u));
                if (rank >= last || rank + __popc(u) <= first) continue;
                for (; u; u &= u - 1, ++rank)
                    if (rank >= first && rank < last) s.col[q][rank - first] = (uint16_t)(w * 32 + __ffs(u) - 1);
            }
        }
        __syncthreads();
        for (int r = tid; r < n[0]; r += TK_THREADS) s.row[r] = (uint16_t)t.loc[s.col[0][r]];
        __syncthreads();
        // ---- 3. stream ----
        const int miss_warps = n[1] == 0 ? 0 : n[0] == 0 ? TK_WARPS : min(TP_MISS_WARPS, (n[1] + TP_U - 1) / TP_U);
        const bool on_misses = warp < miss_warps;
        const int which = on_misses ? 1 : 0;
        const int step = on_misses ? miss_warps : TK_WARPS - miss_warps;
        const char *from = (on_misses ? t.backing : t.arena) + byte_off;
        char *staged = t.arena + (size_t)(t.capacity + lo[1] + r0) * t.row_bytes + byte_off;
        if (on_misses) {
            DIP_TRACE_MIN(t.tr_fetch, 0);
            DIP_TRACE_MIN(t.tr_fetch, 1);
        }
        for (int r1 = on_misses ? warp : warp - miss_warps; r1 < n[which]; r1 += step * TP_U) {
            uint4 q[TP_U];
            float xv[TP_U];
#pragma unroll
            for (int u = 0; u < TP_U; ++u) {
                const int r = r1 + u * step;
                q[u] = make_uint4(0u, 0u, 0u, 0u);
                xv[u] = 0.f;
                if (r < n[which]) {
                    const int col = s.col[which][r], row = on_misses ? col : s.row[r];
                    if (lane_ok) q[u] = __ldcs(reinterpret_cast<const uint4 *>(from + (size_t)row * t.row_bytes));
                    xv[u] = __ldg(p.v + col);
                }
            }
#pragma unroll
            for (int u = 0; u < TP_U; ++u) {
                if (on_misses && lane_ok && r1 + u * step < n[1])
                    *reinterpret_cast<uint4 *>(staged + (size_t)(r1 + u * step) * t.row_bytes) = q[u];
                float w[E];
                decode16<WT>(q[u], w);
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = fmaf(w[e], xv[u], acc[e]);
            }
        }
        if (on_misses) DIP_TRACE_MAX_WARP(t.tr_fetch, 2);
    }
    DIP_TRACE_MAX(p.tr, 3);            // streaming done

    // ---- 4. the warps' sums, pairs first; then the parts', in the last part's CTA (see gemv_fused.cu) ----
#pragma unroll
    for (int e = 0; e < E; ++e) s.red[warp][lane * E + e] = acc[e];
    __syncthreads();
    float sum = 0.f;
    if (tid < SLAB) sum = tree_sum<TK_WARPS>(&s.red[0][tid], 32 * 8);
    if (part != nparts - 1) {
        if (tid < SLAB) mail_put(p.mail + ((size_t)part * p.n_slabs + slab) * SLAB + tid, sum);
    } else {
        if (nparts > 1) {
            const size_t stride = (size_t)p.n_slabs * SLAB;
            float *boxes = p.mail + (size_t)slab * SLAB;
            if (nparts - 1 > MAIL_N) {
                __syncthreads();           // everyone has read s.red
                sum = many_parts<SLAB>(boxes, stride, nparts - 1, sum, &s.red[0][0], t.status, t.wait_limit_ns);
            } else if (tid < SLAB) {
                float a[MAIL_N];
                mail_take<MAIL_N>(boxes + tid, stride, nparts - 1, a, t.status, t.wait_limit_ns);
                ExactSum all(sum);
#pragma unroll
                for (int q = 0; q < MAIL_N; ++q) all.add(a[q]);
                sum = all.value();
            }
        }
        if (tid < SLAB) s.sum[tid] = sum;
        __syncthreads();
        const int j = slab * OUT_PER_SLAB + tid;
        if (tid < OUT_PER_SLAB && j < p.d_out) {
            const int e0 = (tid / C) * 2 * C + (tid % C);     // gate element; its up element is C further
            p.out[j] = WHICH == 0 ? silu_f32(s.sum[e0]) * s.sum[e0 + C] : s.sum[tid];
        }
    }
    // ---- 5. this block's pieces of the staged rows that the cache keeps, into their slots ----
    if (!moves_known(t, &s.go)) return;            // (the barrier inside: all pieces are staged)
    const int32_t *move = t.fetch + 4 + t.staging;
    for (int r1 = lo[1] + warp; r1 < hi[1]; r1 += TK_WARPS * TP_U) {
        int to[TP_U];
        uint4 q[TP_U];
#pragma unroll
        for (int u = 0; u < TP_U; ++u) to[u] = lane_ok && r1 + u * TK_WARPS < hi[1] ? __ldcg(move + r1 + u * TK_WARPS) : -1;
#pragma unroll
        for (int u = 0; u < TP_U; ++u)
            if (to[u] >= 0) q[u] = *reinterpret_cast<const uint4 *>(t.arena + (size_t)(t.capacity + r1 + u * TK_WARPS) * t.row_bytes + byte_off);
#pragma unroll
        for (int u = 0; u < TP_U; ++u)
            if (to[u] >= 0) *reinterpret_cast<uint4 *>(t.arena + (size_t)to[u] * t.row_bytes + byte_off) = q[u];
    }
    DIP_TRACE_MAX(p.tr, 2);
}

TierParams tier_params(dip_ctx *ctx, const dip_tier *t, const dip_cache_update &c)
{
    TierParams p;
    p.d = t->d;
    p.capacity = t->capacity;
    p.staging = t->staging;
    p.row_bytes = t->row_bytes;
    p.mask = c.mask;
    p.split = t->split;
    p.slot = t->slot;
    p.fetch = t->fetch;
    p.loc = t->loc;
    p.backing = (const char *)t->backing;
    p.arena = (char *)t->arena;
    p.counters = t->counters;
    p.cache = c;
    p.moves = ctx->readers + 1;
    p.status = ctx->status;
    p.wait_limit_ns = ctx->block_wait_ns;
    p.tr_book = dip_trace_slot(ctx, 6);
    p.tr_fetch = dip_trace_slot(ctx, 7);
    return p;
}

template <int WT, int WHICH>
dip_status launch_product(dip_ctx *ctx, const TierParams &t, TierProduct &p, int k, cudaStream_t stream)
{
    static_assert(32 * WTraits<WT>::E <= DIP_MAIL_FLOATS, "");
    p.n_slabs = (int)((t.row_bytes + TP_SEG - 1) / TP_SEG);
    p.nparts = row_parts((ctx->sm_count - 1) / p.n_slabs, k, TK_WARPS);       // parts only with one CTA per SM: the mail boxes suffice
    constexpr size_t smem = sizeof(ProductSmem) > sizeof(BookSmem) ? sizeof(ProductSmem) : sizeof(BookSmem);
    static dip_per_device_once once;
    DIP_CUDA_TRY(ctx, dip_raise_smem_limit(once, ctx->device, tier_product_kernel<WT, WHICH>, smem));
    DIP_CUDA_TRY(ctx, dip_launch_pdl(tier_product_kernel<WT, WHICH>, dim3(1 + p.n_slabs * p.nparts), dim3(TK_THREADS), smem, stream, t, p));
    return DIP_OK;
}

// Self-test of waits between blocks that run out: for block 0's word on the moves, and for four sums of a row part, which come after that.
__global__ void __launch_bounds__(TK_THREADS, 1)
tier_waits_selftest_kernel(const TierParams t, float *mail)
{
    __shared__ int go;
    if (threadIdx.x == 0) *t.moves = 0u;
    if (moves_known(t, &go)) atomicExch(t.status, 2);          // (nobody has said anything)
    if (threadIdx.x == 0) {
        float4 a[1];
        mail_take4<1>(mail, 0, 1, a, t.status, t.wait_limit_ns);
        mail_put4(mail, make_float4(1e30f, 1e30f, 1e30f, 1e30f));
    }
}

}  // namespace

dip_status dip_launch_tier_waits_selftest(dip_ctx *ctx, unsigned long long limit_ns, cudaStream_t stream)
{
    TierParams t = {};
    t.moves = ctx->readers + 1;
    t.status = ctx->status;
    t.wait_limit_ns = limit_ns;
    tier_waits_selftest_kernel<<<1, TK_THREADS, 0, stream>>>(t, ctx->mail);
    DIP_CUDA_TRY(ctx, cudaGetLastError());
    return DIP_OK;
}

dip_status dip_launch_tier_product(dip_ctx *ctx, const dip_mlp_weights *w, int which, const dip_tier *t, const dip_cache_update &c,
                                   const float *v, int k, float *out, cudaStream_t stream)
{
    TierProduct p;
    p.d_out = which == 0 ? w->d_ff : w->d_model;
    p.v = v;
    p.out = out;
    p.mail = ctx->mail;
    p.tr = dip_trace_slot(ctx, which == 0 ? 4 : 5);
    const TierParams tp = tier_params(ctx, t, c);
    if (w->wtype == DIP_W_F32)
        return which == 0 ? launch_product<DIP_W_F32, 0>(ctx, tp, p, k, stream) : launch_product<DIP_W_F32, 1>(ctx, tp, p, k, stream);
    return which == 0 ? launch_product<DIP_W_BF16, 0>(ctx, tp, p, k, stream) : launch_product<DIP_W_BF16, 1>(ctx, tp, p, k, stream);
}

dip_status dip_launch_tier_fetch(dip_ctx *ctx, const dip_tier *t, const dip_cache_update &c, cudaStream_t stream)
{
    static_assert(sizeof(BookSmem) + 16 <= 48 * 1024, "");
    DIP_CUDA_TRY(ctx, dip_launch_pdl(tier_fetch_kernel, dim3(DIP_TIER_CTAS), dim3(TK_THREADS), 0, stream, tier_params(ctx, t, c)));
    return DIP_OK;
}
