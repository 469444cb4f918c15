// The column-cache update of Algorithm 1 as a device function for one CTA of 1024 threads: the whole of
// cache_update_kernel, and the blocks without rows beside a product's.
#pragma once

#include "select_core.cuh"

namespace {

// c' = cache_update(c, m) of Algorithm 1 with the LRU policy of Sec. 5.1 (or LFU when use counters are
// given), from the mask bits and the state alone.  One CTA: it runs beside a product that fills the
// other SMs, and a chain of exchanges between CTAs would cost more than the few thousand columns an SM
// has to look at.
// A warp owns NB consecutive blocks of 128 columns, a lane four consecutive columns of each (one
// 16-byte load and one 16-byte store), and what lies in between never goes through shared memory (64 registers
// do not hold all of it in the wider variants: 416 bytes of spill stores in cache_update_kernel, which stay in L1).  The eviction
// key of a column that may be evicted (resident and outside the mask) is the age of its last use
// (LFU: t + 1 - uses), of any other column 0.
// Bound by the SM's issue rate and its trips through shared memory.  Alone, LRU, after 38 updates:
// 7.9 us at d = 17920 (load 1.5, histogram 2.1 + search 0.7, ties 1.2, stamps 2.1), 4.4 us at 5120;
// one column per lane swept four times through shared memory with 4-byte stores took 14.4 and 6.6 us.
//
// mask_bits and stamp_now (the stamps as they are) may lie in shared memory.  s.hist and small[] are zero on
// entry (cache_update_clear), though not yet synchronised.  poll() is called by the last warp (which seldom has
// columns) some time before may_write(), which all threads call before the first stamp is written (and which is a
// barrier unless it always says yes); if it says no, the state is left as it was.  (The counters, which only this
// function reads, are written before that, and restored.)
constexpr int CU_SPREAD = 8;                            // copies of the counters of the small digits,
constexpr int CU_SMALL = 256;                           // which nearly all keys have: ages of a few updates

__device__ __forceinline__ void cache_update_clear(TkShared &s, unsigned int *small)
{
    const int tid = threadIdx.x;
    s.hist[2 * tid] = s.hist[2 * tid + 1] = 0;
    small[2 * tid] = small[2 * tid + 1] = 0;
}

// The counters as they were before the uses of this mask (out of line: only after a wait that ran out).
__device__ __noinline__ void take_uses_back(const uint32_t *mask_bits, int d, int32_t *count)
{
    for (int c = threadIdx.x; c < d; c += TK_THREADS)
        if ((mask_bits[c >> 5] >> (c & 31)) & 1u) --count[c];
}

template <int NB, bool LFU, typename Poll, typename MayWrite>
__device__ __forceinline__ void block_cache_update(const uint32_t *mask_bits, int d, const int32_t *stamp_now, int32_t *stamp,
                                                   int32_t *count, int32_t *meta, int capacity, TkShared &s, unsigned int *small,
                                                   const Poll &poll, const MayWrite &may_write)
{
    static_assert(CU_SMALL * CU_SPREAD == 2 * TK_THREADS && RADIX_BINS == 2 * TK_THREADS, "two counters per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_res = meta[0];
    const int t_now = meta[1] + 1;
    const int col0 = warp * (NB * 128) + lane * 4;      // this lane's first column; block i is 128 i further

    // ---- the state and the mask: eviction keys ----
    uint32_t ek[NB][4];
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
                const int4 q = *reinterpret_cast<const int4 *>(stamp_now + c);
                st[i][0] = q.x; st[i][1] = q.y; st[i][2] = q.z; st[i][3] = q.w;
                if (LFU) {
                    const int4 n = *reinterpret_cast<const int4 *>(count + c);
                    cn[i][0] = n.x; cn[i][1] = n.y; cn[i][2] = n.z; cn[i][3] = n.w;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (c + e < d) {
                        st[i][e] = stamp_now[c + e];
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
                ek[i][e] = st[i][e] >= 0 && !((nib >> e) & 1u) ? (uint32_t)(t_now - (LFU ? cn[i][e] : st[i][e])) & 0x7fffffffu : 0u;
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
    const uint32_t misses = keep & ~res;

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
            unsigned int *mine = small + (lane & (CU_SPREAD - 1));
            while (hi > 0) {
                const int w = hi < RADIX_BITS ? hi : RADIX_BITS, shift = hi - w;
                const uint32_t digit_mask = (1u << w) - 1u;
                if (t_now < CU_SMALL) {
                    // (one pass, and every digit is a small one)
#pragma unroll
                    for (int i = 0; i < NB; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (ek[i][e]) atomicAdd(mine + (ek[i][e] & (CU_SMALL - 1)) * CU_SPREAD, 1u);
                } else {
#pragma unroll
                    for (int i = 0; i < NB; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (ek[i][e] != 0u && (ek[i][e] & prefix_mask) == prefix) {
                                const uint32_t dg = (ek[i][e] >> shift) & digit_mask;
                                atomicAdd(dg < CU_SMALL ? mine + dg * CU_SPREAD : &s.hist[dg], 1u);
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
                    cache_update_clear(s, small);
                    __syncthreads();
                }
            }
            T2 = prefix;
            quota2 = krem;
        }
    }
    if (warp == TK_WARPS - 1) poll();
    // ---- if only the first quota2 ties go: the ties in front of each warp, and inside the one warp in
    //      which the quota runs out, in front of each lane.  Likewise the misses, if some find no room ----
    uint32_t ties = 0u;
    if (quota2 > 0 && T2 != 0u) {
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (ek[i][e] == T2) ties |= 1u << (4 * i + e);
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
    if (!may_write()) {
        if (LFU) take_uses_back(mask_bits, d, count);
        return;
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int c = col0 + 128 * i;
        uint32_t gone = (ties >> (4 * i)) & 0xfu;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (ek[i][e] > T2) gone |= 1u << e;
        const uint32_t used = (use >> (4 * i)) & 0xfu;
        if (!(gone | used)) continue;
        if (c + 4 <= d) {
            int4 v = *reinterpret_cast<const int4 *>(stamp_now + c);
            v.x = gone & 1u ? -1 : used & 1u ? t_now : v.x;
            v.y = gone & 2u ? -1 : used & 2u ? t_now : v.y;
            v.z = gone & 4u ? -1 : used & 4u ? t_now : v.z;
            v.w = gone & 8u ? -1 : used & 8u ? t_now : v.w;
            *reinterpret_cast<int4 *>(stamp + c) = v;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (((gone | used) >> e) & 1u) stamp[c + e] = (gone >> e) & 1u ? -1 : t_now;
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
}

// The same in the variant for d columns, whose state lies in registers.
template <typename Poll, typename MayWrite>
__device__ __forceinline__ void block_cache_update_any(const uint32_t *mask_bits, int d, const int32_t *stamp_now, int32_t *stamp,
                                                       int32_t *count, int32_t *meta, int capacity, TkShared &s, unsigned int *small,
                                                       const Poll &poll, const MayWrite &may_write)
{
    const auto run = [&](auto nb) {
        constexpr int NB = decltype(nb)::value;
        if (count) block_cache_update<NB, true>(mask_bits, d, stamp_now, stamp, count, meta, capacity, s, small, poll, may_write);
        else block_cache_update<NB, false>(mask_bits, d, stamp_now, stamp, count, meta, capacity, s, small, poll, may_write);
    };
    static_assert(DIP_MAX_D <= 8 * 128 * TK_WARPS, "");
    if (d <= 2 * 128 * TK_WARPS) run(Int<2>());
    else if (d <= 5 * 128 * TK_WARPS) run(Int<5>());
    else run(Int<8>());
}

}  // namespace
