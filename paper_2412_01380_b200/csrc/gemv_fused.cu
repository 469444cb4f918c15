// One token, F32 / BF16 weights: a product kernel that builds its own mask.
//
// In a step, each product (Eq. 1-3) needs the top-k mask of its input (Eq. 7-8, or the cache-aware
// ranking of Algorithm 1), and a select kernel in front of it costs a kernel boundary, the mask's
// trip through global memory, and a device that idles while one CTA selects.  The select by one
// 15-bit histogram (select_core.cuh) is short enough for every CTA of the product to run it for
// itself - same code, same inputs, hence the same rows everywhere, with nothing to wait for -
// and to go straight on to its rows.  The kept set is the stand-alone select's, bit for bit.
//
// Memory is idle until the first row is asked for, so what lies between the threshold's bin and that
// moment is kept short: the columns above the bin ("sure") go from the flags in registers into the
// CTA's row list with one block-wide prefix sum, and the bin's few dozen columns ("ties") are ranked
// by one warp while the others already stream.  What bounds these phases is the number of instructions, as
// all 32 warps issue them (1200 per warp, 9600 of a scheduler's cycles, when each key was tested by itself and
// each warp searched the histogram).  List order: sure columns, then the kept ties by rank; a CTA owns a
// 512-byte segment of the packed rows and a share of that list (32 warps x 4 loads in flight).  Its sums
// meet in a fixed order: warps in shared memory, row parts in the CTA of the last part, which the others
// send theirs to.
//
// The updates of column caches ride along with the last down product of a call, as blocks without rows
// (UPD).  The down input's own cache is among them: its block makes the mask together with the others and
// writes the cache's state once all of them have read it.  Other launches do without that code, which would
// cost each of them 1.3 us (block_f32 shapes, 14.3 against 16.9 us per step of two launches).
#include <math.h>
#include <string.h>

#include <type_traits>

#include "cache_update.cuh"
#include "gemv_common.cuh"

namespace {

constexpr int GF_SEG = 512;
constexpr int GF_NW = TK_THREADS / 32;     // 32 warps
constexpr int GF_U = 4;                    // loads in flight per lane
constexpr double GF_AHEAD_BYTES = 15e6;        // rows asked for once the threshold's bin is known: gate/up,
constexpr double GF_AHEAD_MORE_BYTES = 12e6;   // gate/up that has asked for some before,
constexpr double GF_AHEAD_DOWN_BYTES = 16e6;   // down,
constexpr double GF_EARLY_BYTES = 25e6;        // and before that (see `early`)
constexpr size_t GF_SMEM_LIMIT = (size_t)224 * 1024;   // dynamic shared memory a launch may ask for

struct FusedParams {
    // product
    const char *W;
    size_t row_bytes;
    int d_in, d_out;
    int n_slabs, nparts;
    int ahead, ahead_of;         // the rows of how many groups of columns out of how many (the parts together) are asked for as soon
                                 // as the threshold's bin is known; see there
    int early;                   // gate/up, chained: of how many groups before that, if their keys are larger than
    uint32_t sure;               // this: rms is 1, so fewer than k columns can be larger than sqrt(d / k) (times gamma, where that is above 1)
    uint32_t by_prod, by_ahead;  // ceil(2^32 / n), n = blocks with rows; ahead_of
    int x_near;                  // gate/up: room in shared memory for the values of x
    float *out;
    float *mail;                 // [nparts][n_slabs][segment elements]; DIP_MAIL_EMPTY outside a launch
    int *status;
    unsigned long long wait_limit_ns;
    unsigned long long *tr;
    uint16_t *key_coarse;        // gate/up: top 16 bits of the rank keys of h (nullptr: not wanted)
    const int32_t *key_stamp;
    float key_gamma;
    // select
    const float *xa;             // gate/up: x, or the previous layer's x when xb is given; down: h
    const float *xb;             // gate/up, chained: the previous layer's y
    float *x_out;                // gate/up, chained: where CTA 0 writes x = (xa + xb) / rms(xa + xb)
    const uint16_t *coarse;      // down: top 16 bits of the rank keys of h
    int k;
    float gamma;
    const int32_t *stamp;        // cache state of this input (CA) or unused
    uint32_t *mask_out;
};

struct FusedUpdates {            // UPD
    unsigned int *readers;       // CTAs that have read the stamps; zero between launches
    dip_cache_update own;        // this input's cache (its mask is made here)
    dip_cache_updates beside;    // caches that nothing in the launch depends on
};

struct __align__(16) FusedSmem {
    TkFine fine;                           // the select's histogram; afterwards the warps' sums [32][segment elements]
                                           // and, in its second half, their partial sums [1024]
    TkShared ts;
    unsigned int maskw[DIP_MAX_D / 32];    // the mask (in the CTA that writes it, and under heavy ties)
    int wsum[GF_NW];
    uint16_t tie[TK_TIE_LIMIT];            // the kept columns of the threshold's bin, by rank
    int go;                                // UPD: all have read the stamps
};
static_assert(GF_NW * 32 * 8 <= TK_FINE_WORDS / 2 && TK_THREADS <= TK_FINE_WORDS / 2, "the sums fit the histogram");

// Ranks [lo, hi) of the rows in `words` (a bit set in shared memory, complete and visible) as a list
// in idx[].  One word per thread (DIP_MAX_D / 32 words at most); all threads call it; ends with a
// barrier.  (Heavy ties only: otherwise the list is built from the flags in registers.)
__device__ __forceinline__ void list_rows(FusedSmem &s, const unsigned int *words, int mask_words, int lo, int hi,
                                          uint16_t *idx)
{
    static_assert(DIP_MAX_D / 32 <= TK_THREADS, "one mask word per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t u = tid < mask_words ? words[tid] : 0u;
    const int c = __popc(u);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) s.wsum[warp] = incl;
    __syncthreads();
    int total;
    int rank = warp_array_prefix(s.wsum, warp, lane, total) + incl - c;
    for (; u; u &= u - 1, ++rank)
        if (rank >= lo && rank < hi) idx[rank - lo] = (uint16_t)(tid * 32 + __ffs(u) - 1);
    __syncthreads();
}

// The sure columns (c of them flagged by this thread) whose rank among them lies in [lo, hi) to idx[], in the
// order of the warps, their lanes, and the flags of put(emit)'s calls emit(base, flags, bit, column).
// Deterministic, which is all that is asked of the order.  All threads call it; the barrier inside also
// publishes what was written before the call; does not end with one.
template <typename Put>
__device__ __forceinline__ void list_sure(FusedSmem &s, int c, int lo, int hi, uint16_t *idx, const Put &put)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) s.wsum[warp] = incl;
    __syncthreads();
    const int at = (int)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)s.wsum[lane] : 0u) + incl - c - lo;   // list place of the first
    const unsigned n = (unsigned)(hi - lo);
    // (every flag finds its place by itself: a walk from one set bit to the next is a chain of latencies)
    if (at < hi - lo && at + c > 0)
        put(at, [&](int base, uint32_t flags, int bit, int col) {
            const unsigned place = (unsigned)(base + __popc(flags & ((1u << bit) - 1u)));
            if (((flags >> bit) & 1u) && place < n) idx[place] = (uint16_t)col;
        });
}

// acc += sum over rows idx[first], idx[first + stride], ... below n_rows of row segment x value,
// U rows in flight per lane.
template <int WT>
__device__ __forceinline__ void stream_rows(const uint16_t *idx, int first, int stride, int n_rows, const char *base,
                                            size_t row_bytes, bool lane_ok, const float *xsrc,
                                            float (&acc)[WTraits<WT>::E])
{
    constexpr int E = WTraits<WT>::E;
    for (int r0 = first; r0 < n_rows; r0 += stride * GF_U) {
        uint4 q[GF_U];
        float xv[GF_U];
#pragma unroll
        for (int u = 0; u < GF_U; ++u) {
            const int r = r0 + u * stride;
            q[u] = make_uint4(0u, 0u, 0u, 0u);
            xv[u] = 0.f;
            if (r < n_rows) {
                const int i = idx[r];
                if (lane_ok) q[u] = __ldcs(reinterpret_cast<const uint4 *>(base + (size_t)i * row_bytes));
                xv[u] = xsrc[i];
            }
        }
#pragma unroll
        for (int u = 0; u < GF_U; ++u) {
            float w[E];
            decode16<WT>(q[u], w);
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] = fmaf(w[e], xv[u], acc[e]);
        }
    }
}

// Block part * n_slabs + slab owns segment `slab`, row part `part`.  UPD: then come the blocks without rows, one
// for each cache of u.beside, and last the one that completes the mask and updates this input's cache.  NQ =
// chunks of columns per thread (gate/up: 4 columns each, down: 8).  AHEAD: rows are asked for ahead.  Dynamic shared memory: FusedSmem, then d_in
// words (rounded up to four: the CTA's row list; the updating block's copy of the stamps; under heavy ties the rank
// keys before that), then for gate/up (x_near) the d_in values of x.  Shared memory is kept small: what it does not
// take is L1, which the rows in flight pass through (with the 72 KB of h beside the rest, 224 KB in all, the down
// product of 17920 dense rows took 11 us longer).
template <int WT, int WHICH, bool CA, bool NORM, int NQ, bool UPD, bool AHEAD>
__global__ void __launch_bounds__(TK_THREADS, 1)
gemv_fused_kernel(const FusedParams p, const std::conditional_t<UPD, FusedUpdates, Int<0>> u)
{
    constexpr int E = WTraits<WT>::E;
    constexpr int SLAB = 32 * E;
    constexpr int OUT_PER_SLAB = WHICH == 0 ? SLAB / 2 : SLAB;
    constexpr int W = WHICH == 0 ? 4 : 8;
    static_assert(WTraits<WT>::C == E, "a lane's elements are all gate or all up, the next lane's their partners");
    static_assert(!UPD || (CA && WHICH == 1), "updates ride with a down product that has a cache");
    extern __shared__ __align__(16) unsigned char dyn[];
    FusedSmem &s = *reinterpret_cast<FusedSmem *>(dyn);
    const int dpad = (p.d_in + 3) & ~3;
    uint32_t *keys = reinterpret_cast<uint32_t *>(dyn + sizeof(FusedSmem));
    uint16_t *idx = reinterpret_cast<uint16_t *>(keys);
    float *xs = reinterpret_cast<float *>(keys + dpad);

    DIP_TRACE_MIN(p.tr, 0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slab = (int)blockIdx.x % p.n_slabs, part = (int)blockIdx.x / p.n_slabs, nparts = p.nparts;
    const int n_prod = p.n_slabs * nparts;
    const bool updater = UPD && blockIdx.x == gridDim.x - 1;
    const bool writer = UPD ? updater : (int)blockIdx.x == n_prod - 1;   // writes the mask (the last part ranks the ties anyway)
    const int mask_words = (p.d_in + 31) >> 5;
    const size_t byte_off = (size_t)slab * GF_SEG + lane * 16;
    const bool lane_ok = byte_off < p.row_bytes;
    // this part's share of the k rows (part * k fits 32 bits: at most one part per SM, at most DIP_MAX_D rows)
    const int lo = updater ? p.k : (int)((unsigned)part * (unsigned)p.k / (unsigned)nparts);
    const int hi = updater ? p.k : (int)((unsigned)(part + 1) * (unsigned)p.k / (unsigned)nparts);
    const bool every = p.k == p.d_in;                         // nothing to select
    // position tid of a segment's sums (see below) is element `el`; gate/up: of output `o` if it is a gate element
    const int el = E == 8 ? ((tid & 127) >> 2) * 8 + (tid >> 7) * 4 + (tid & 3) : tid;
    const int o = WHICH == 0 ? (el / (2 * E)) * E + el % E : el;
    const int j_out = slab * OUT_PER_SLAB + o;
    const bool out_ok = tid < SLAB && (WHICH == 1 || ((tid >> 2) & 1) == 0) && j_out < p.d_out;

    bool staged = false;                                       // updater: keys[] is a copy of the stamps
    if constexpr (UPD) {
        if ((int)blockIdx.x >= n_prod) {
            // (small[], like the select's histogram that lies there otherwise, and the counters)
            if (!updater) cache_update_clear(s.ts, s.fine.hist);
            else if (!every) fine_zero(s.fine);
            dip_grid_dependency_wait();
            dip_launch_dependents();
            if (!updater) {
                const dip_cache_update &c = u.beside.at[(int)blockIdx.x - n_prod];
                block_cache_update_any(c.mask, c.d, c.stamp, c.stamp, c.count, c.meta, c.capacity, s.ts, s.fine.hist, []() {},
                                       []() { return true; });
                return;
            }
            // the stamps on their way to shared memory while the mask is made: once the other CTAs stream, a trip to
            // global memory takes several microseconds
            for (int q = tid; q < p.d_in / 4; q += TK_THREADS)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(keys + 4 * q)), "l"(p.stamp + 4 * q) : "memory");
            staged = true;
        }
    }
    if (!updater) {
        if (!every) fine_zero(s.fine);
        dip_grid_dependency_wait();
        DIP_TRACE_MIN(p.tr, 1);
        dip_launch_dependents();
    }

    // the stamp that the epilogue's rank key needs travels while the rows stream
    int key_stamp = 0;
    if (WHICH == 0 && p.key_coarse && p.key_stamp && out_ok) key_stamp = __ldcg(p.key_stamp + j_out);

    // (rows asked for ahead are shared out over the blocks: this one's are those of groups q of columns with q % n_prod its index)
    const auto mine = [&](int q) { return q - (int)__umulhi((unsigned)q, p.by_prod) * n_prod == (int)blockIdx.x; };

    // ---- the rank keys of the input and their histogram, in every CTA ----
    const int n_q = p.d_in / W;
    // groups of the threads before this one: the list has the threads' columns in thread order
    const int before = tid * (n_q / TK_THREADS) + min(tid, n_q % TK_THREADS);
    uint32_t kk[NQ][4];                    // gate/up: full keys of four columns; down: 16-bit keys of eight
    if constexpr (WHICH == 0) {
        // one trip to memory for x (or the two vectors that make it) and the stamps
        float4 r[NQ];
        int4 st[NQ];
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const int q = tid + j * TK_THREADS;
            r[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            st[j] = make_int4(0, 0, 0, 0);
            if (q < n_q) {
                r[j] = reinterpret_cast<const float4 *>(p.xa)[q];
                if (CA) st[j] = reinterpret_cast<const int4 *>(p.stamp)[q];
                if (NORM) {
                    const float4 vb = reinterpret_cast<const float4 *>(p.xb)[q];
                    r[j] = make_float4(r[j].x + vb.x, r[j].y + vb.y, r[j].z + vb.z, r[j].w + vb.w);
                }
            }
        }
        float scale = 1.0f;
        if (NORM) {
            // 1 / rms, summed in block_residual_scale's order
            float ss = 0.f;
#pragma unroll
            for (int j = 0; j < NQ; ++j)
                if (tid + j * TK_THREADS < n_q) {
                    ss = fmaf(r[j].x, r[j].x, ss);
                    ss = fmaf(r[j].y, r[j].y, ss);
                    ss = fmaf(r[j].z, r[j].z, ss);
                    ss = fmaf(r[j].w, r[j].w, ss);
                }
            scale = block_rms_scale(ss, p.d_in, s.ts.wf, &s.ts.scale);
        } else {
            __syncthreads();               // histogram zeroed
        }
        float *x_out = NORM && blockIdx.x == 0 ? p.x_out : nullptr;
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const int q = tid + j * TK_THREADS;
            if (q < n_q) {
                if (NORM) r[j] = make_float4(r[j].x * scale, r[j].y * scale, r[j].z * scale, r[j].w * scale);
                if (x_out) reinterpret_cast<float4 *>(x_out)[q] = r[j];
                if (NORM || p.x_near) reinterpret_cast<float4 *>(xs)[q] = r[j];
                kk[j][0] = rank_key<CA>(r[j].x, st[j].x, p.gamma);
                kk[j][1] = rank_key<CA>(r[j].y, st[j].y, p.gamma);
                kk[j][2] = rank_key<CA>(r[j].z, st[j].z, p.gamma);
                kk[j][3] = rank_key<CA>(r[j].w, st[j].w, p.gamma);
                if (AHEAD && NORM && before < p.early && mine(q)) {
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (kk[j][t] > p.sure) l2_prefetch(p.W + (size_t)(4 * q + t) * p.row_bytes, (unsigned)p.row_bytes);
                }
                if (!every) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) fine_count_hi(s.fine, kk[j][t]);
                }
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const int q = tid + j * TK_THREADS;
            if (q < n_q && !every) {
                const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(p.coarse) + q);
                kk[j][0] = v.x; kk[j][1] = v.y; kk[j][2] = v.z; kk[j][3] = v.w;
            }
        }
        __syncthreads();                   // histogram zeroed
#pragma unroll
        for (int j = 0; j < NQ; ++j)
            if (tid + j * TK_THREADS < n_q && !every) {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    fine_count_lo(s.fine, kk[j][t]);
                    fine_count_hi(s.fine, kk[j][t]);
                }
            }
    }

    // ---- this part's rows: n_list of them in idx[], and ranks tie_lo .. tie_hi - 1 of the ties in s.tie ----
    int n_list = hi - lo, tie_lo = 0, tie_hi = 0;
    int krem = 0, n_c = 0;
    if (every) {
        for (int r = tid; r < n_list; r += TK_THREADS) idx[r] = (uint16_t)(lo + r);
        if (writer)
            for (int w = tid; w < mask_words; w += TK_THREADS) s.maskw[w] = 0xffffffffu;
        __syncthreads();
    } else {
        __syncthreads();
        fine_find(s.fine, s.ts, p.k);
        const uint32_t b = (uint32_t)s.ts.bcast[0];
        krem = s.ts.bcast[1];
        n_c = s.ts.bcast[2];
        // Rows of each part on their way to L2 while the list is made: whole rows, and of chained gate/up inputs the surely kept ones
        // before that.  As many as come in that time; what is still under way when the first rows are waited for delays them.  Three
        // Phi-3-Medium blocks, graph, us: none at all 111; gate/up only, 15 MB 108; with up to 25 MB before that 105; and 16 MB for
        // down 104.  Gate/up: the first rows of each part.  Down: of the threads as if they had equally many groups each, which
        // is some way into the list for most parts (at their very starts: one step of 5120 / 17920 33.0 us, 32.7 like this)
        const unsigned at = (unsigned)((WHICH == 0 ? before : tid) * nparts);
        if (AHEAD && at - __umulhi(at, p.by_ahead) * p.ahead_of < (unsigned)p.ahead) {
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const int q = tid + j * TK_THREADS;
                if (q < n_q && mine(q)) {
#pragma unroll
                    for (int t = 0; t < W; ++t) {
                        bool ask;
                        if constexpr (WHICH == 0) ask = kk[j][t] > ((b << 16) | 0xffffu) && !(NORM && before < p.early && kk[j][t] > p.sure);
                        else ask = ((kk[j][t >> 1] >> (16 * (t & 1))) & 0xffffu) > b;
                        if (ask) l2_prefetch(p.W + (size_t)(W * q + t) * p.row_bytes, (unsigned)p.row_bytes);
                    }
                }
            }
        }
        if (n_c > TK_TIE_LIMIT) {
            // masses of equal keys: the general select on full keys
            if (staged) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                staged = false;
            }
            __syncthreads();
            if constexpr (WHICH == 0) {
#pragma unroll
                for (int j = 0; j < NQ; ++j)
                    if (tid + j * TK_THREADS < n_q)
                        *reinterpret_cast<uint4 *>(keys + 4 * (tid + j * TK_THREADS)) = make_uint4(kk[j][0], kk[j][1], kk[j][2], kk[j][3]);
            } else {
                for (int e = tid; e < p.d_in; e += TK_THREADS) keys[e] = rank_key<CA>(p.xa[e], CA ? p.stamp[e] : 0, p.gamma);
            }
            __syncthreads();
            general_select(keys, p.d_in, p.k, s.ts, s.maskw);
            __syncthreads();
            list_rows(s, s.maskw, mask_words, lo, hi, idx);
            n_c = 0;
        } else {
            // Columns above the bin: flags gt; the bin's columns: candidates (in any order).  Flag bit of column
            // t of a group: gate/up: t; down, whose keys are compared two at a time (the top bit of each half
            // survives the subtraction where the key is no smaller): 12 + t / 2, in the upper half for odd t
            uint32_t gt[NQ], eqs[NQ];
            int c_gt = 0, c_eq = 0;
            const uint32_t above = (b << 16) | 0xffffu;       // a full key above the bin is larger than this
            const uint32_t ge1 = (b + 1) * 0x10001u, ge0 = b * 0x10001u;
            constexpr uint32_t TOP = 0x80008000u;
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                gt[j] = eqs[j] = 0u;
                const int q = tid + j * TK_THREADS;
                if (q < n_q) {
                    uint32_t eq = 0u;
                    if constexpr (WHICH == 0) {
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            if (kk[j][t] > above) gt[j] |= 1u << t;
                            if (kk[j][t] >= (b << 16)) eq |= 1u << t;
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const uint32_t w = kk[j][t] | TOP;
                            gt[j] |= ((w - ge1) & TOP) >> (3 - t);
                            eq |= ((w - ge0) & TOP) >> (3 - t);
                        }
                    }
                    eqs[j] = eq & ~gt[j];
                    c_gt += __popc(gt[j]);
                    c_eq += __popc(eqs[j]);
                }
                if (writer && (tid & ~31) + j * TK_THREADS < n_q) {      // (the whole warp or none of it)
                    constexpr int LANES = 32 / W;                        // lanes per mask word
                    uint32_t w = gt[j];
                    if (WHICH == 1) {
                        w = 0u;
#pragma unroll
                        for (int t = 0; t < 8; ++t) w |= ((gt[j] >> (12 + t / 2 + 16 * (t & 1))) & 1u) << t;
                    }
                    w <<= W * (lane % LANES);
#pragma unroll
                    for (int m = 1; m < LANES; m <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, m);
                    if (lane % LANES == 0 && q < n_q) s.maskw[q / LANES] = w;
                }
            }
            if (c_eq) {
                int slot = atomicAdd(&s.fine.n_cand, c_eq);
#pragma unroll
                for (int j = 0; j < NQ; ++j)
                    for (uint32_t eq = eqs[j]; eq; eq &= eq - 1, ++slot) {
                        const int f = __ffs(eq) - 1, t = WHICH == 0 ? f : 2 * (f & 3) + (f >> 4);
                        s.fine.cand[slot] = (uint16_t)(W * (tid + j * TK_THREADS) + t);
                        if (WHICH == 0) s.fine.ckey[slot] = t == 0 ? kk[j][0] : t == 1 ? kk[j][1] : t == 2 ? kk[j][2] : kk[j][3];
                    }
            }
            const int n_sure = p.k - krem;
            n_list = max(0, min(hi, n_sure) - lo);
            tie_lo = max(lo, n_sure) - n_sure;
            tie_hi = max(hi, n_sure) - n_sure;
            list_sure(s, c_gt, lo, hi, idx, [&](int base, const auto &emit) {
#pragma unroll
                for (int j = 0; j < NQ; ++j) {
                    if (j * TK_THREADS >= n_q) break;
#pragma unroll
                    for (int t = 0; t < W; ++t)
                        emit(base, gt[j], WHICH == 0 ? t : 12 + t / 2 + 16 * (t & 1), W * (tid + j * TK_THREADS) + t);
                    base += __popc(gt[j]);
                }
            });
            __syncthreads();
        }
    }

    const bool ranks = n_c > 0 && (tie_lo < tie_hi || writer);
    const auto tie_key = [&](int col, int c) {
        return WHICH == 0 ? s.fine.ckey[c] : rank_key<CA>(__ldcg(p.xa + col), CA ? __ldcg(p.stamp + col) : 0, p.gamma);
    };
    if constexpr (UPD) {
        if (updater) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            if (ranks && warp == 0) rank_ties(s.fine, n_c, krem, s.tie, s.maskw, tie_key);
            __syncthreads();
            for (int w = tid; w < mask_words; w += TK_THREADS) p.mask_out[w] = s.maskw[w];
            cache_update_clear(s.ts, s.fine.hist);
            // The stamps may change once every block with rows has read them.  Blocks start in index order and this is
            // the last one, so all the others are running or done
            block_cache_update_any(
                s.maskw, p.d_in, staged ? reinterpret_cast<const int32_t *>(keys) : p.stamp, u.own.stamp, u.own.count, u.own.meta,
                u.own.capacity, s.ts, s.fine.hist,
                [&]() {
                    if (lane == 0) {
                        s.go = wait_count(u.readers, (unsigned)n_prod, p.status, p.wait_limit_ns);
                        *u.readers = 0u;                       // ready for the next launch
                    }
                },
                [&]() {
                    __syncthreads();
                    return s.go != 0;
                });
            DIP_TRACE_MAX(p.tr, 2);
            return;
        }
    }

    // ---- stream.  Where this CTA ranks ties, warp 0 does that first, takes their rows, and gets so many fewer of
    //      the listed ones ----
    const float *xsrc = WHICH == 0 && (NORM || p.x_near) ? xs : p.xa;
    const char *base = p.W + byte_off;
    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    int n_even = n_list;                                       // rows shared out over all warps
    if (ranks) {
        n_even = min(n_list, max(0, (n_list + tie_hi - tie_lo) / GF_NW - (tie_hi - tie_lo) - GF_U) * GF_NW);
        if (warp == 0) {
            rank_ties(s.fine, n_c, krem, s.tie, writer ? s.maskw : nullptr, tie_key);
            if constexpr (UPD) {
                if (lane == 0) count_one(u.readers);
            }
            stream_rows<WT>(s.tie, tie_lo, 1, tie_hi, base, p.row_bytes, lane_ok, xsrc, acc);
        }
    } else if constexpr (UPD) {
        if (tid == 0) count_one(u.readers);                    // (the stamps were read before the last barrier)
    }
    stream_rows<WT>(idx, warp, GF_NW, n_even, base, p.row_bytes, lane_ok, xsrc, acc);
    if (warp > 0 && n_even < n_list)
        stream_rows<WT>(idx, n_even + warp - 1, GF_NW - 1, n_list, base, p.row_bytes, lane_ok, xsrc, acc);
    DIP_TRACE_MAX(p.tr, 3);            // streaming done

    // ---- the warps' sums, in warp order.  Element e of lane l lies at position (e / 4) * 128 + 4 l + e % 4 ----
    float *red = reinterpret_cast<float *>(s.fine.hist), *psum = red + TK_FINE_WORDS / 2;
#pragma unroll
    for (int h = 0; h < E / 4; ++h)
        *reinterpret_cast<float4 *>(red + warp * SLAB + h * 128 + lane * 4) =
            make_float4(acc[4 * h], acc[4 * h + 1], acc[4 * h + 2], acc[4 * h + 3]);
    __syncthreads();
    constexpr int G = TK_THREADS / SLAB;                       // threads per position
    {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < GF_NW / G; ++w) t += red[((tid / SLAB) * (GF_NW / G) + w) * SLAB + tid % SLAB];
        psum[tid] = t;
    }
    if (writer)
        for (int w = tid; w < mask_words; w += TK_THREADS) p.mask_out[w] = s.maskw[w];
    __syncthreads();
    const size_t stride = (size_t)p.n_slabs * SLAB;
    float *boxes = p.mail + (size_t)slab * SLAB;
    float others = 0.f;
    if (nparts - 1 > MAIL_N && part == nparts - 1)
        others = mail_sum_wide<SLAB, TK_THREADS>(boxes, stride, nparts - 1, red, p.status, p.wait_limit_ns);
    if (tid >= SLAB) return;
    float t = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) t += psum[g * SLAB + tid];
    // ---- the parts, in part order, in the last part's CTA.  A sum is its own message: the CTA that adds them up
    //      waits until none of its inputs is "empty" any more, and empties them for the next launch.  Blocks start
    //      in index order and only the last ones wait, so what they wait for is running or done ----
    if (nparts > 1) {
        if (part != nparts - 1) {
            mail_put(boxes + (size_t)part * stride + tid, t);
            DIP_TRACE_MAX(p.tr, 2);
            return;
        }
        if (nparts - 1 <= MAIL_N) others = mail_sum(boxes + tid, stride, nparts - 1, p.status, p.wait_limit_ns);
        t = others + t;
    }
    // ---- epilogue ----
    const float up = __shfl_down_sync(0xffffffffu, t, 4);      // gate/up: a gate element's up element is four positions on
    if (out_ok) {
        const float r = WHICH == 0 ? silu_f32(t) * up : t;
        p.out[j_out] = r;
        if (WHICH == 0 && p.key_coarse) {
            // what the select would form from h_j and the stamp, cut to its top 16 bits
            float a = fabsf(r);
            if (p.key_stamp) a = __fmul_rn(a, key_stamp >= 0 ? 1.0f : p.key_gamma);
            p.key_coarse[j_out] = (uint16_t)((__float_as_uint(a) & 0x7fffffffu) >> 16);
        }
    }
    DIP_TRACE_MAX(p.tr, 2);
}

template <int WT, int WHICH, bool CA, bool NORM, int NQ, bool UPD, bool AHEAD>
dip_status launch_fused_as(dip_ctx *ctx, const FusedParams &p, const std::conditional_t<UPD, FusedUpdates, Int<0>> &u, int extra,
                           size_t smem, cudaStream_t stream)
{
    static dip_per_device_once once;
    const auto kernel = gemv_fused_kernel<WT, WHICH, CA, NORM, NQ, UPD, AHEAD>;
    DIP_CUDA_TRY(ctx, dip_raise_smem_limit(once, ctx->device, kernel, GF_SMEM_LIMIT));
    DIP_CUDA_TRY(ctx, dip_launch_pdl(kernel, dim3(p.n_slabs * p.nparts + extra), dim3(TK_THREADS), smem, stream, p, u));
    return DIP_OK;
}

// (launches that ask for no rows ahead do without that code: 2048 / 8192, BF16, keep ratio 0.1, steps with other weights each, 13.6 us with it and 13.1 without)
template <int WT, int WHICH, bool CA, bool NORM, int NQ, bool UPD>
dip_status launch_fused(dip_ctx *ctx, const FusedParams &p, const std::conditional_t<UPD, FusedUpdates, Int<0>> &u, int extra,
                        size_t smem, cudaStream_t stream)
{
    return p.ahead ? launch_fused_as<WT, WHICH, CA, NORM, NQ, UPD, true>(ctx, p, u, extra, smem, stream)
                   : launch_fused_as<WT, WHICH, CA, NORM, NQ, UPD, false>(ctx, p, u, extra, smem, stream);
}

// Columns per thread: a row's keys stay in registers, so the variant for wide inputs (which spills) only takes
// what the narrow one cannot.
template <int WT, bool CA, bool NORM>
dip_status launch_fused_gate_up(dip_ctx *ctx, const FusedParams &p, size_t smem, cudaStream_t stream)
{
    if (p.d_in <= 2 * 4 * TK_THREADS) return launch_fused<WT, 0, CA, NORM, 2, false>(ctx, p, Int<0>(), 0, smem, stream);
    return launch_fused<WT, 0, CA, NORM, TK_VEC_ITERS, false>(ctx, p, Int<0>(), 0, smem, stream);
}

template <int WT>
dip_status launch_fused_wt(dip_ctx *ctx, const FusedParams &p, int which, bool ca, bool norm, const FusedUpdates *u,
                           size_t smem, cudaStream_t stream)
{
    if (which == 0) {
        if (ca) return norm ? launch_fused_gate_up<WT, true, true>(ctx, p, smem, stream)
                            : launch_fused_gate_up<WT, true, false>(ctx, p, smem, stream);
        return norm ? launch_fused_gate_up<WT, false, true>(ctx, p, smem, stream)
                    : launch_fused_gate_up<WT, false, false>(ctx, p, smem, stream);
    }
    constexpr int NQ = TK_COARSE_ITERS;
    if (u) return launch_fused<WT, 1, true, false, NQ, true>(ctx, p, *u, u->beside.n + 1, smem, stream);
    return ca ? launch_fused<WT, 1, true, false, NQ, false>(ctx, p, Int<0>(), 0, smem, stream)
              : launch_fused<WT, 1, false, false, NQ, false>(ctx, p, Int<0>(), 0, smem, stream);
}

size_t fused_smem_bytes(int d_in, bool x_near)
{
    const size_t dpad = ((size_t)d_in + 3) & ~(size_t)3;
    return sizeof(FusedSmem) + dpad * 4 + (x_near ? dpad * 4 : 0);
}

// Segments and row parts of a launch of k rows; false when the shape does not fit this path.
bool fused_plan(const dip_ctx *ctx, const dip_mlp_weights *w, int which, bool norm, int k, FusedParams &p)
{
    if (!ctx->gemv_direct || !ctx->fuse_select) return false;
    if (w->wtype != DIP_W_F32 && w->wtype != DIP_W_BF16) return false;
    p.d_in = which == 0 ? w->d_model : w->d_ff;
    p.d_out = which == 0 ? w->d_ff : w->d_model;
    if (which == 1 && ((p.d_in & 31) != 0 || p.d_in > 8 * TK_COARSE_ITERS * TK_THREADS)) return false;
    p.x_near = which == 0 && fused_smem_bytes(p.d_in, true) <= GF_SMEM_LIMIT;
    if ((norm && !p.x_near) || fused_smem_bytes(p.d_in, false) > GF_SMEM_LIMIT) return false;
    const size_t row_elems = which == 0 ? (size_t)2 * w->d_ff : (size_t)w->d_model;
    p.row_bytes = w->wtype == DIP_W_F32 ? row_elems * 4 : row_elems * 2;
    p.n_slabs = (int)((p.row_bytes + GF_SEG - 1) / GF_SEG);
    // one CTA per SM, and where that is cheap two SMs to spare for the blocks that update caches
    int most = ctx->sm_count / p.n_slabs;              // (DIP_MAIL_FLOATS per SM suffice)
    if (most > 4 && most * p.n_slabs > ctx->sm_count - 2) most = (ctx->sm_count - 2) / p.n_slabs;
    p.nparts = row_parts(most, k, GF_NW);
    return true;
}

// Self-test of the waits between blocks.  Block 0 collects ten row parts of which one is missing, and sends that one too
// late; block 1 updates a cache whose readers (two are expected) have not all counted, and the missing one counts too late.
__global__ void __launch_bounds__(TK_THREADS, 1)
block_waits_selftest_kernel(float *mail, unsigned int *readers, int *status, unsigned long long limit_ns, const dip_cache_update c)
{
    constexpr int SLAB = 256, N = MAIL_N + 2, MISSING = MAIL_N;
    __shared__ TkShared ts;
    __shared__ __align__(16) unsigned int small[CU_SMALL * CU_SPREAD];
    __shared__ float sum[TK_THREADS];
    __shared__ int go;
    const int tid = threadIdx.x;
    if (blockIdx.x == 0) {
        if (tid < SLAB)
            for (int q = 0; q < N; ++q)
                if (q != MISSING) mail_put(mail + q * SLAB + tid, 1.f);
        (void)mail_sum_wide<SLAB, TK_THREADS>(mail, SLAB, N, sum, status, limit_ns);
        if (tid < SLAB) mail_put(mail + MISSING * SLAB + tid, 1e30f);
        return;
    }
    cache_update_clear(ts, small);
    block_cache_update_any(
        c.mask, c.d, c.stamp, c.stamp, c.count, c.meta, c.capacity, ts, small,
        [&]() {
            if (tid % 32 == 0) {
                count_one(readers);
                go = wait_count(readers, 2u, status, limit_ns);
                *readers = 0u;
            }
        },
        [&]() {
            __syncthreads();
            return go != 0;
        });
    if (tid == TK_THREADS - 32) count_one(readers);
}

}  // namespace

dip_status dip_launch_block_waits_selftest(dip_ctx *ctx, unsigned long long limit_ns, const dip_cache_update &c, cudaStream_t stream)
{
    block_waits_selftest_kernel<<<2, TK_THREADS, 0, stream>>>(ctx->mail, ctx->readers, ctx->status, limit_ns, c);
    DIP_CUDA_TRY(ctx, cudaGetLastError());
    return DIP_OK;
}

int dip_gemv_fused_update_room(const dip_ctx *ctx, const dip_mlp_weights *w, int k)
{
    FusedParams p;
    // (a wave of products that fills the SMs to the last one leaves none)
    return fused_plan(ctx, w, 1, false, k, p) ? (ctx->sm_count - p.n_slabs * p.nparts % ctx->sm_count) % ctx->sm_count : 0;
}

bool dip_gemv_fused_supported(const dip_ctx *ctx, const dip_mlp_weights *w, int which, bool norm)
{
    if (w->wtype == DIP_W_INT4_G128) return dip_gemv_int4_selects(ctx, w, which);
    FusedParams p;
    return fused_plan(ctx, w, which, norm, 1, p);
}

dip_status dip_launch_gemv_fused(dip_ctx *ctx, const dip_mlp_weights *w, int which, const dip_fused_select *sel,
                                 float *out, cudaStream_t stream, dip_gemv_keys *keys)
{
    const bool norm = which == 0 && sel->xb != nullptr;
    if (w->wtype == DIP_W_INT4_G128) {
        const size_t row_elems = which == 0 ? (size_t)2 * w->d_ff : (size_t)w->d_model;
        GemvParams g = {};
        g.W = (const char *)(which == 0 ? w->gate_up : w->down);
        g.row_bytes = row_elems / 2;
        g.scales = (const uint16_t *)(which == 0 ? w->gate_up_scales : w->down_scales);
        g.scale_row_elems = row_elems;
        g.v = sel->xa;                                  // (down; gate/up keeps x in shared memory)
        g.d_in = which == 0 ? w->d_model : w->d_ff;
        g.d_out = which == 0 ? w->d_ff : w->d_model;
        g.mask_words = (g.d_in + 31) / 32;
        g.out = out;
        g.batch = 1;
        g.mail = ctx->mail;
        g.status = ctx->status;
        g.tr = dip_trace_slot(ctx, which == 0 ? 4 : 5);
        g.key_gamma = 1.0f;
        if (keys) keys->written = 0;
        if (which == 0 && keys && keys->coarse) {
            g.key_coarse = keys->coarse;
            g.key_stamp = keys->stamp;
            g.key_gamma = keys->gamma;
            keys->written = 1;
        }
        return dip_launch_gemv_int4(ctx, g, which, sel->k, 0, sel, stream);
    }
    FusedParams p;
    if (!fused_plan(ctx, w, which, norm, sel->k, p)) return DIP_ERR_UNSUPPORTED;
    p.W = (const char *)(which == 0 ? w->gate_up : w->down);
    p.out = out;
    p.mail = ctx->mail;
    p.status = ctx->status;
    p.wait_limit_ns = ctx->block_wait_ns;
    p.tr = dip_trace_slot(ctx, which == 0 ? 4 : 5);
    p.key_coarse = nullptr;
    p.key_stamp = nullptr;
    p.key_gamma = 1.0f;
    if (keys) keys->written = 0;
    if (which == 0 && keys && keys->coarse) {
        p.key_coarse = keys->coarse;
        p.key_stamp = keys->stamp;
        p.key_gamma = keys->gamma;
        keys->written = 1;
    }
    // Whether rows are asked for ahead, and how many.  Gate/up: from 8 MB on, all rows if there are no more (less gains nothing: keep
    // ratio 0.1 of 2048 / 8192, 6.7 MB).  One step, BF16, each with other weights: 3072 / 8192 with 10 MB 14.37 us without and 13.9
    // with, 4096 / 11008 with 18 MB 16.3 and 16.1; F32 2048 / 5632, 23 MB, 15.9 with 15 MB and 16.6 with 20.  The surely kept rows before
    // that from 20 MB on (3072 / 8192, 25 MB, twelve chained blocks 19.0 us a block without and 18.6 with; 17 MB 16.5 either way) and from
    // a fifth of the columns kept: of a tenth, few are that large.  Down: from 32 MB on (22 MB, 4096 / 11008, step 23.6 us without
    // and 24.0 with; 46 MB, 5120 / 17920, 32.9 and 32.3).  Where every column is kept nothing is searched for (three dense blocks of
    // 4096 / 11008 181.8 us with rows asked for early, 179.4 without)
    const int n_q = p.d_in / (which == 0 ? 4 : 8);
    const double bytes = (double)p.row_bytes * sel->k;
    const bool early = norm && bytes > 20e6 && 5 * (long long)sel->k >= p.d_in;
    const double ahead = which == 1 ? GF_AHEAD_DOWN_BYTES : early ? GF_AHEAD_MORE_BYTES : GF_AHEAD_BYTES;
    const double from = which == 1 ? 2 * GF_AHEAD_DOWN_BYTES : 8e6;
    p.ahead_of = which == 1 && n_q > TK_THREADS ? TK_THREADS : n_q;
    p.by_ahead = (uint32_t)((0x100000000ull + (unsigned)p.ahead_of - 1) / (unsigned)p.ahead_of);
    p.ahead = bytes > from && sel->k < p.d_in ? (int)(p.ahead_of * (ahead < bytes ? ahead / bytes : 1.0)) : 0;
    // (of Laplace or Student-t inputs a quarter of the kept columns are that large, hence the quarter)
    p.early = 0;
    if (early && p.ahead) p.early = GF_EARLY_BYTES < bytes / 4 ? (int)(n_q * GF_EARLY_BYTES / (bytes / 4)) : n_q;
    // (a gamma of 64 and nothing resident, two blocks of 4096 / 11008 at keep ratio 0.25: 63.8 us where every row with a key above
    // sqrt(d / k) was asked for, 52.9 with gamma 1)
    const float sure = sqrtf((float)p.d_in / (float)sel->k) * 1.001f * (sel->stamp ? fmaxf(1.0f, sel->gamma) : 1.0f);
    memcpy(&p.sure, &sure, sizeof(sure));
    p.by_prod = (uint32_t)((0x100000000ull + (unsigned)(p.n_slabs * p.nparts) - 1) / (unsigned)(p.n_slabs * p.nparts));
    p.xa = sel->xa;
    p.xb = sel->xb;
    p.x_out = sel->x_out;
    p.coarse = sel->coarse;
    p.k = sel->k;
    p.gamma = sel->gamma;
    p.stamp = sel->stamp;
    p.mask_out = sel->mask_out;
    const size_t smem = fused_smem_bytes(p.d_in, p.x_near);
    FusedUpdates u;
    if (sel->update) {
        u.readers = ctx->readers;
        u.own = dip_update_of(sel->update, nullptr);
        u.beside.n = 0;
        if (sel->beside) u.beside = *sel->beside;
    }
    const FusedUpdates *up = sel->update ? &u : nullptr;
    return w->wtype == DIP_W_F32 ? launch_fused_wt<DIP_W_F32>(ctx, p, which, sel->stamp != nullptr, norm, up, smem, stream)
                                 : launch_fused_wt<DIP_W_BF16>(ctx, p, which, sel->stamp != nullptr, norm, up, smem, stream);
}
