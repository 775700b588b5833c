// tpx_general.cu -- the general (global-memory) path: tpx_decode,
// tpx_cluster, tpx_centroid, the exact redo of a tpx_process call whose
// input the fused kernel cannot hold on chip, and the streaming calls.
//
// decode  : tile aggregates of the two unwrap chains (Sec. IV.A) -> prefix
//           over tiles -> per-packet unwrapped times and the trigger list ->
//           each pixel binned to the most recent trigger in time by binary
//           search, cut at tof_max (Sec. IV.B), timewalk table subtracted
//           (Sec. IV.C) -> kept pixels compacted in stream order.
// cluster : stable LSD radix sort of the hits on (shot, corrected ToF) --
//           ties keep stream order. In that order a gap larger than dt ends
//           every cluster, so the sorted hits split into independent
//           segments. One warp clusters a segment of up to 64 hits in
//           registers: a compact one from a grid of cells, any other by ballots
//           that give each hit's adjacency row (Sec. V.A box rule) and
//           local-maximum flag (Sec. V.B); components are closures over the
//           rows seeded at the earliest hit; the root's int64 moments are warp
//           sums. Up to 256 hits one block does it in shared memory. Longer
//           segments (shots whose particles arrive within dt of each other)
//           find their pairs through a hash of (shot, x, y) cells and join them
//           in a global lock-free union-find whose root is the smallest position.
// centroid: records in ascending label order (root flags counted per block in
//           stream order), f64 final division (Sec. V.C); PAPER mode sums the
//           box neighbourhood of each local maximum.
// No capacity limit besides 2^31 - 1 kept pixels per call.
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <vector>

#include "tpx.h"
#include "tpx_common.cuh"
#include "tpx_ctx.h"
#include "tpx_fused.cuh"
#include "tpx_unwrap.cuh"

namespace tpxg {

using namespace tpxk;

constexpr int GT = 256;             // threads per block
constexpr int GW = GT / 32;
constexpr int GK = 16;              // packets (or keys) per thread
constexpr int GTILE = GT * GK;      // 4096
constexpr int kBias = 32768;        // corrected ToF + bias >= 0 for int16 timewalk shifts

// ------------------------------------------------------------ block scans
__device__ GAgg block_scan_agg_g(const GAgg &v, GAgg *s_w, GAgg *total, long long tp, long long tt) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    GAgg incl = warp_incl_scan(v, lane, tp, tt);
    GAgg wex = shfl_up_agg(incl, 1);
    if (lane == 0) wex = agg_id();
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    if (w == 0) {
        GAgg x = lane < GW ? s_w[lane] : agg_id();
        GAgg xi = warp_incl_scan(x, lane, tp, tt);
        GAgg xe = shfl_up_agg(xi, 1);
        if (lane == 0) xe = agg_id();
        if (lane < GW) s_w[lane] = xe;
        if (lane == GW - 1) *total = xi;
    }
    __syncthreads();
    GAgg r = acomb(s_w[w], wex, tp, tt);
    __syncthreads();
    return r;
}

__device__ long long block_scan_ll(long long v, long long *s_w, long long *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    if (w == 0) {
        long long x = lane < GW ? s_w[lane] : 0;
        long long xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += u;
        }
        if (lane < GW) s_w[lane] = xi - x;
        if (lane == GW - 1) *total = xi;
    }
    __syncthreads();
    long long r = s_w[w] + incl - v;
    __syncthreads();
    return r;
}

// single-block scans (PT threads, each over a contiguous strip of items)
constexpr int PT = 1024;
__device__ long long block_excl_ll_pt(long long v, long long *s32, long long *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s32[w] = incl;
    __syncthreads();
    if (w == 0) {
        const long long x = s32[lane];
        long long xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += u;
        }
        s32[lane] = xi - x;
        if (lane == 31) *total = xi;
    }
    __syncthreads();
    const long long r = s32[w] + incl - v;
    __syncthreads();
    return r;
}
__device__ GAgg block_excl_agg_pt(const GAgg &v, GAgg *s32, long long tp, long long tt) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const GAgg incl = warp_incl_scan(v, lane, tp, tt);
    GAgg lex = shfl_up_agg(incl, 1);
    if (lane == 0) lex = agg_id();
    if (lane == 31) s32[w] = incl;
    __syncthreads();
    if (w == 0) {
        const GAgg xi = warp_incl_scan(s32[lane], lane, tp, tt);
        GAgg xe = shfl_up_agg(xi, 1);
        if (lane == 0) xe = agg_id();
        s32[lane] = xe;
    }
    __syncthreads();
    const GAgg r = acomb(s32[w], lex, tp, tt);
    __syncthreads();
    return r;
}
__device__ __forceinline__ void strip_of(long long items, long long *b, long long *e) {
    const long long per = (items + PT - 1) / PT;
    *b = min(items, (long long)threadIdx.x * per);
    *e = min(items, *b + per);
}

// the block's flags: a warp takes 32 * GK consecutive items, 32 per ballot;
// returns the slot of the warp's first flagged item within the block
template <class F>
__device__ __forceinline__ unsigned block_flags(long long n, F flag, unsigned (&m)[GK], unsigned *s_c, unsigned *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long base = blockIdx.x * (long long)GTILE + w * (32 * GK) + lane;
    unsigned f = 0, c = 0;
#pragma unroll
    for (int j = 0; j < GK; ++j) {   // no ballot yet: the loads of all rounds are in flight together
        const long long i = base + 32 * j;
        if (i < n && flag(i, j)) f |= 1u << j;
    }
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        m[j] = __ballot_sync(0xffffffffu, (f >> j) & 1u);
        c += __popc(m[j]);
    }
    if (lane == 0) s_c[w] = c;
    __syncthreads();
    unsigned before = 0, all = 0;
#pragma unroll
    for (int k = 0; k < GW; ++k) {
        before += k < w ? s_c[k] : 0u;
        all += s_c[k];
    }
    *total = all;
    return before;
}

// ------------------------------------------------------------ decode kernels
// a tile's chain aggregates, its triggers, and whether a wrap step of either
// stream lies inside it: a warp per 512 packets, its loads ahead of its steps
__global__ void __launch_bounds__(GT) k_tile_agg(const uint64_t *pk, long long n, long long tp, long long tt,
                                                 GAgg *tagg, long long *tcnt, unsigned char *twrap) {
    __shared__ GAgg s_a[32];
    __shared__ bool s_wrap[GW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long tile = blockIdx.x, base = tile * GTILE;
    const int cnt = (int)min((long long)GTILE, n - base), per = GTILE / GW;
    const int qb = w * per, qe = min(cnt, qb + per);
    WarpPart<4> part;
    if (qb < qe) part.run(pk + base, (reinterpret_cast<uintptr_t>(pk) & 15) == 0, qb, qe, tp, tt, lane);
    GAgg a;
    GChain head;
    part.result(&a, &head);
    const bool wraps = part.wraps || __any_sync(0xffffffffu, part.tdc_wraps);   // (opposite steps: a sum of 0)
    if (lane == 0) {
        s_a[w] = a;
        s_wrap[w] = wraps;
    }
    __syncthreads();
    if (w == 0) {
        const GAgg mine = lane < GW ? s_a[lane] : agg_id();
        const GAgg incl = warp_incl_scan(mine, lane, tp, tt);
        const bool wrap = __any_sync(0xffffffffu, lane < GW && s_wrap[lane]);
        if (lane == 31) {
            tagg[tile] = incl;
            tcnt[tile] = incl.tdc.n;
        }
        GAgg before = shfl_up_agg(incl, 1);
        if (lane == 0) before = agg_id();
        const bool step = (before.pix.n && mine.pix.n && jump(mine.pix.first - before.pix.last, tp) != 0) ||
                          (before.tdc.n && mine.tdc.n && jump(mine.tdc.first - before.tdc.last, tt) != 0);
        const bool any = __any_sync(0xffffffffu, step);
        if (lane == 0) twrap[tile] = wrap || any;
    }
}

// exclusive prefix over tiles, starting from the state before the call (one
// block: strips of tiles, a block scan of the strip aggregates, then strips)
__global__ void __launch_bounds__(PT) k_tile_prefix(const GAgg *tagg, GAgg *tpre, const long long *tcnt, long long *toff,
                                                    long long tiles, long long tp, long long tt, long long *n_trig_out,
                                                    const GAgg *E0, GAgg *state_out) {
    __shared__ GAgg s_a[32];
    __shared__ long long s_c[32];
    __shared__ long long s_tot;
    long long b, e;
    strip_of(tiles, &b, &e);
    GAgg a = agg_id();
    long long cn = 0;
    for (long long t = b; t < e; ++t) {
        a = acomb(a, tagg[t], tp, tt);
        cn += tcnt[t];
    }
    const GAgg ex = block_excl_agg_pt(a, s_a, tp, tt);
    long long off = block_excl_ll_pt(cn, s_c, &s_tot);
    GAgg acc = acomb(E0 ? *E0 : agg_id(), ex, tp, tt);
    for (long long t = b; t < e; ++t) {
        tpre[t] = acc;
        toff[t] = off;
        acc = acomb(acc, tagg[t], tp, tt);
        off += tcnt[t];
    }
    if (threadIdx.x == PT - 1) {   // its strip is the last (possibly empty) one
        toff[tiles] = off;
        *n_trig_out = off;
        if (state_out) *state_out = acc;
    }
}

// A tile without a wrap step (nearly all) adds one constant per stream: warps
// read and write 512 consecutive packets each, bound by the bytes. The others
// follow the chains packet by packet.
__global__ void __launch_bounds__(GT) k_unwrap(const uint64_t *pk, long long n, const GAgg *tagg, const GAgg *tpre,
                                               const unsigned char *twrap, const long long *toff,
                                               long long tp, long long tt, long long *t_all, long long *trig,
                                               long long trig_cap, unsigned *status, long long *trig_pos) {
    __shared__ GAgg s_w[GW];
    __shared__ GAgg s_tot;
    __shared__ unsigned s_c[GW];
    const long long tile = blockIdx.x, base = tile * GTILE;
    const GAgg before = tpre[tile], own = tagg[tile];
    const bool wraps = twrap[tile] || (before.pix.n && own.pix.n && jump(own.pix.first - before.pix.last, tp) != 0) ||
                       (before.tdc.n && own.tdc.n && jump(own.tdc.first - before.tdc.last, tt) != 0);
    if (!wraps) {
        const int lane = threadIdx.x & 31;
        const long long q0 = base + (threadIdx.x >> 5) * (32 * GK) + lane;
        const long long dp = before.pix.sum * kPixPeriod, dd = before.tdc.sum * kTdcPeriod;
        uint64_t v[GK];
#pragma unroll
        for (int j = 0; j < GK; ++j) v[j] = q0 + 32 * j < n ? pk[q0 + 32 * j] : 0;
        unsigned m[GK], total;
        unsigned o = block_flags(n, [&](long long, int j) { return (unsigned)(v[j] >> 60) == 0x6u; }, m, s_c, &total);
#pragma unroll
        for (int j = 0; j < GK; ++j) {
            const long long q = q0 + 32 * j;
            const unsigned h = (unsigned)(v[j] >> 60);
            long long t = 0;
            if (h == 0xBu) t = pix_raw(v[j]) + dp;
            else if (h == 0x6u) {
                t = tdc_raw(v[j]) + dd;
                const long long ti = toff[tile] + o + __popc(m[j] & ((1u << lane) - 1u));
                if (ti < trig_cap) {
                    trig[ti] = t;
                    if (trig_pos) trig_pos[ti] = q;
                } else {
                    atomicOr(status, ST_TRIG_CAP);
                }
            }
            o += __popc(m[j]);
            if (q < n) t_all[q] = t;
        }
        return;
    }
    const long long q0 = base + threadIdx.x * GK;
    GAgg a = agg_id();
    for (int j = 0; j < GK; ++j) {
        const long long q = q0 + j;
        if (q >= n) break;
        const uint64_t w = pk[q];
        const unsigned h = (unsigned)(w >> 60);
        if (h == 0xBu) chain_push(a.pix, pix_raw(w), tp);
        else if (h == 0x6u) chain_push(a.tdc, tdc_raw(w), tt);
    }
    const GAgg ex = block_scan_agg_g(a, s_w, &s_tot, tp, tt);
    const GAgg st = acomb(tpre[tile], ex, tp, tt);
    bool hp = st.pix.n > 0, ht = st.tdc.n > 0;
    long long lp = st.pix.last, ep = st.pix.sum, lt = st.tdc.last, et = st.tdc.sum;
    long long ti = toff[tile] + ex.tdc.n;
    for (int j = 0; j < GK; ++j) {
        const long long q = q0 + j;
        if (q >= n) break;
        const uint64_t w = pk[q];
        const unsigned h = (unsigned)(w >> 60);
        long long t = 0;
        if (h == 0xBu) {
            const long long r = pix_raw(w);
            if (hp) ep += jump(r - lp, tp);
            hp = true;
            lp = r;
            t = r + ep * kPixPeriod;
        } else if (h == 0x6u) {
            const long long r = tdc_raw(w);
            if (ht) et += jump(r - lt, tt);
            ht = true;
            lt = r;
            t = r + et * kTdcPeriod;
            if (ti < trig_cap) {
                trig[ti] = t;
                if (trig_pos) trig_pos[ti] = q;
            } else {
                atomicOr(status, ST_TRIG_CAP);
            }
            ++ti;
        }
        t_all[q] = t;
    }
}

// the trigger count of the call, or -1 when it exceeded the trigger capacity
// (the status is latched and nothing is binned)
__device__ __forceinline__ long long usable_triggers(const long long *n_trig, long long trig_cap) {
    const long long v = *n_trig;
    return v > trig_cap ? -1 : v;
}

__global__ void k_check_trig(const long long *trig, const long long *n_trig, long long trig_cap, unsigned *status) {
    const long long ntr = usable_triggers(n_trig, trig_cap);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i + 1 < ntr; i += (long long)gridDim.x * blockDim.x)
        if (trig[i + 1] < trig[i]) atomicOr(status, ST_TRIG_ORDER);
}

// most recent trigger in time: last index with trig <= t, or -1
__device__ __forceinline__ long long shot_of(const long long *trig, long long ntr, long long t) {
    long long lo = 0, hi = ntr;
    while (lo < hi) {
        const long long mid = lo + ((hi - lo) >> 1);
        if (trig[mid] <= t) lo = mid + 1; else hi = mid;
    }
    return lo - 1;
}

// per tile: kept pixels and the drop counters; per packet: its shot, or -1 when
// it is not a kept pixel. A thread's packets follow one another in time, so the
// shot of the one before is tried first; a search over the triggers for the rest.
__global__ void __launch_bounds__(GT) k_bin(const uint64_t *pk, long long n, const long long *t_all, const long long *trig,
                                            const long long *n_trig, long long trig_cap, long long tof_max, int *shot,
                                            long long *tile_kept, unsigned long long *counters) {
    __shared__ unsigned s_c[6];
    const long long tile = blockIdx.x, base = tile * GTILE;
    const long long ntr = usable_triggers(n_trig, trig_cap);
    if (threadIdx.x < 6) s_c[threadIdx.x] = 0;
    __syncthreads();
    unsigned keep = 0, bg = 0, pre = 0, pix = 0, tdc = 0, bad = 0;
    long long s = -1, from = 1, to = 0;   // the last pixel's shot and its times [from, to)
    constexpr int B = 8;   // packets whose loads are in flight together
    for (int j0 = 0; j0 < GK && ntr >= 0; j0 += B) {
        unsigned h[B];
        long long t[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const long long q = base + (j0 + j) * GT + threadIdx.x;
            h[j] = q < n ? (unsigned)(pk[q] >> 60) : 0x100u;
            t[j] = q < n ? t_all[q] : 0;
        }
#pragma unroll
        for (int j = 0; j < B; ++j) {
            if (h[j] == 0x100u) break;
            int out = -1;
            if (h[j] == 0xBu) {
                ++pix;
                if (t[j] < from || t[j] >= to) {
                    s = shot_of(trig, ntr, t[j]);
                    from = s >= 0 ? trig[s] : LLONG_MIN;
                    to = s + 1 < ntr ? trig[s + 1] : LLONG_MAX;
                }
                if (s < 0) ++pre;
                else if (t[j] - from > tof_max) ++bg;
                else {
                    ++keep;
                    out = (int)s;
                }
            } else if (h[j] == 0x6u) ++tdc;
            else ++bad;
            shot[base + (j0 + j) * GT + threadIdx.x] = out;
        }
    }
    const unsigned vals[6] = {keep, bg, pre, pix, tdc, bad};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const unsigned v = __reduce_add_sync(0xffffffffu, vals[k]);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_c[k], v);
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int idx[6] = {C_KEPT, C_DROP_BG, C_DROP_PRE, C_PIXELS, C_TDCS, C_CORRUPT};
        if (s_c[threadIdx.x]) atomicAdd(&counters[idx[threadIdx.x]], (unsigned long long)s_c[threadIdx.x]);
        if (threadIdx.x == 0) tile_kept[tile] = s_c[0];
    }
}

// exclusive prefix of per-tile counts (one block)
__global__ void __launch_bounds__(PT) k_count_prefix(const long long *cnt, long long *off, long long tiles,
                                                     long long *total_out) {
    __shared__ long long s_c[32];
    __shared__ long long s_tot;
    long long b, e;
    strip_of(tiles, &b, &e);
    long long v = 0;
    for (long long t = b; t < e; ++t) v += cnt[t];
    long long o = block_excl_ll_pt(v, s_c, &s_tot);
    for (long long t = b; t < e; ++t) {
        off[t] = o;
        o += cnt[t];
    }
    if (threadIdx.x == PT - 1) {
        off[tiles] = o;
        if (total_out) *total_out = o;
    }
}

// kept pixels in stream order (a warp takes 512 consecutive packets, so its
// writes are runs)
__global__ void __launch_bounds__(GT) k_compact(const uint64_t *pk, long long n, long long idx_base, const long long *t_all,
                                                const long long *trig, const long long *n_trig, long long trig_cap,
                                                const int *shot, const int16_t *lut, const long long *tile_off,
                                                tpx_hits hits, long long cap, unsigned *status, const GAgg *E0) {
    __shared__ unsigned s_c[GW];
    const long long trig_base = E0 ? E0->tdc.n : 0;
    if (usable_triggers(n_trig, trig_cap) < 0) return;
    const int lane = threadIdx.x & 31;
    const long long tile = blockIdx.x;
    const long long q0 = tile * GTILE + (threadIdx.x >> 5) * (32 * GK) + lane;
    int sh[GK];
#pragma unroll
    for (int j = 0; j < GK; ++j) sh[j] = q0 + 32 * j < n ? shot[q0 + 32 * j] : -1;
    unsigned m[GK], total;
    const unsigned before = block_flags(n, [&](long long, int j) { return sh[j] >= 0; }, m, s_c, &total);
    long long o = tile_off[tile] + before;
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        if (sh[j] >= 0) {
            const long long q = q0 + 32 * j, slot = o + __popc(m[j] & ((1u << lane) - 1u));
            if (slot < cap) {
                const uint64_t w = pk[q];
                const long long t = t_all[q];
                const int tot = pix_tot(w);
                const long long corr = lut ? (long long)lut[tot] : 0LL;
                hits.index[slot] = idx_base + q;
                hits.shot[slot] = sh[j] + trig_base;
                hits.t[slot] = t - corr;
                hits.tof[slot] = (int32_t)(t - trig[sh[j]] - corr);
                hits.x[slot] = (uint8_t)pix_x(w);
                hits.y[slot] = (uint8_t)pix_y(w);
                hits.tot[slot] = (uint16_t)tot;
            } else {
                atomicOr(status, ST_CLUSTER_CAP);
            }
        }
        o += __popc(m[j]);
    }
}

// ------------------------------------------------------------ radix sort
// Stable LSD sort of (key, value) pairs on 8-bit digits, in tiles of 4096 keys;
// per digit: each tile's histogram (the first digit's is taken while the keys
// are made), a scan of them over the tiles, and the placing. A CTA ranks its
// tile in registers (a warp's 32 keys by eight ballots, its own counters in
// shared memory), puts it in digit order in shared memory and writes runs. Keys
// of 32 bits where (shot, ToF) fits them.
// What bounds it: instruction issue (the ranking) on large inputs, the launches
// on small ones. Measured per digit of 6.0e6 / 1.2e6 hits: 109 / 45 us with a
// scatter of 16 rounds, each waiting for the one before, and three scan
// launches; 60 / 19 us with one launch whose tiles look back for the counts
// before them (their polling took two thirds of the issue slots); now 58 / 17.
template <class K>
__device__ __forceinline__ unsigned digit_of(K key, int shift) { return (unsigned)(key >> shift) & 255u; }
// one count in shared memory; a warp whose keys share the digit, as those of
// the upper digits do, adds once. act: the lanes that call.
__device__ __forceinline__ void count_digit(unsigned *h, unsigned d, unsigned act) {
    int same = 0;
    __match_all_sync(act, d, &same);
    if (!same) atomicAdd(&h[d], 1u);
    else if ((int)(threadIdx.x & 31) == __ffs(act) - 1) atomicAdd(&h[d], (unsigned)__popc(act));
}
template <class K>
__global__ void __launch_bounds__(GT) k_digit_hist(const K *keys, long long n, int shift, unsigned *hist) {
    __shared__ unsigned s_h[256];
    s_h[threadIdx.x] = 0;
    const long long base = blockIdx.x * (long long)GTILE + threadIdx.x;
    K k[GK];
#pragma unroll
    for (int j = 0; j < GK; ++j) k[j] = base + j * GT < n ? keys[base + j * GT] : K(0);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        const bool ok = base + j * GT < n;
        const unsigned act = __ballot_sync(0xffffffffu, ok);
        if (ok) count_digit(s_h, digit_of(k[j], shift), act);
    }
    __syncthreads();
    hist[blockIdx.x * 256ll + threadIdx.x] = s_h[threadIdx.x];
}
// per digit the exclusive prefix over the tiles, in place, and the total: a CTA
// takes 32 digits, each of its warps a stretch of the tiles
__global__ void __launch_bounds__(PT) k_digit_scan(unsigned *hist, long long tiles, unsigned *total) {
    __shared__ unsigned s_sum[32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long per = (tiles + 31) / 32, t0 = min(tiles, w * per), t1 = min(tiles, t0 + per);
    unsigned *h = hist + blockIdx.x * 32 + lane;
    unsigned sum = 0;
#pragma unroll 8
    for (long long t = t0; t < t1; ++t) sum += h[t * 256];
    s_sum[w][lane] = sum;
    __syncthreads();
    unsigned run = 0, all = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const unsigned v = s_sum[k][lane];
        run += k < w ? v : 0u;
        all += v;
    }
    if (w == 0) total[blockIdx.x * 32 + lane] = all;
    for (long long t = t0; t < t1; t += 8) {
        unsigned v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = t + k < t1 ? h[(t + k) * 256] : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (t + k < t1) h[(t + k) * 256] = run;
            run += v[k];
        }
    }
}
template <class K>
__global__ void __launch_bounds__(GT, sizeof(K) == 4 ? 4 : 3) k_digit_place(const K *kin, const unsigned *vin, long long n,
                                                                           int shift, const unsigned *offs,
                                                                           const unsigned *total, K *kout, unsigned *vout) {
    extern __shared__ __align__(16) unsigned char s_buf[];   // the tile in digit order: keys, values
    __shared__ unsigned s_wh[GW][256];      // per warp: digit counts, then the warp's first slot of each digit
    __shared__ unsigned s_off[256];         // output position of a digit's run minus its slot in the tile
    __shared__ long long s_w[GW];
    __shared__ long long s_tot;
    K *bk = reinterpret_cast<K *>(s_buf);
    unsigned *bv = reinterpret_cast<unsigned *>(s_buf + GTILE * sizeof(K));
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const long long base = blockIdx.x * (long long)GTILE;
    const int valid = (int)min((long long)GTILE, n - base);
    const int i0 = w * (32 * GK) + lane;
    K key[GK];
    unsigned pos[GK];
#pragma unroll
    for (int j = 0; j < GK; ++j) key[j] = i0 + 32 * j < valid ? kin[base + i0 + 32 * j] : ~K(0);   // past the end: behind every key
    const unsigned before = offs[blockIdx.x * 256ll + t], all = total[t];   // thread t: digit t
#pragma unroll
    for (int k = 0; k < GW; ++k) s_wh[k][t] = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        const unsigned d = digit_of(key[j], shift);
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
            peers &= ((d >> b) & 1u) ? m : ~m;
        }
        const int leader = __ffs(peers) - 1;
        unsigned old = 0;
        if (lane == leader) {
            old = s_wh[w][d];
            s_wh[w][d] = old + __popc(peers);
        }
        pos[j] = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    unsigned cnt = 0;
#pragma unroll
    for (int k = 0; k < GW; ++k) {
        const unsigned x = s_wh[k][t];
        s_wh[k][t] = cnt;
        cnt += x;
    }
    // the digits' starts in the whole output and in the tile, one scan
    const long long both = block_scan_ll(((long long)all << 16) | cnt, s_w, &s_tot);
    const unsigned lstart = (unsigned)(both & 0xFFFF);
    s_off[t] = (unsigned)(both >> 16) + before - lstart;
#pragma unroll
    for (int k = 0; k < GW; ++k) s_wh[k][t] += lstart;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        const int i = i0 + 32 * j;
        const unsigned q = pos[j] + s_wh[w][digit_of(key[j], shift)];
        bk[q] = key[j];
        bv[q] = i < valid ? (vin ? vin[base + i] : (unsigned)(base + i)) : 0u;
    }
    __syncthreads();
#pragma unroll 4
    for (int i = t; i < valid; i += GT) {
        const K k = bk[i];
        const unsigned g = s_off[digit_of(k, shift)] + i;
        kout[g] = k;
        vout[g] = bv[i];
    }
}

// exclusive scan of block counts in place (one block)
__global__ void __launch_bounds__(PT) k_scan_bsum(unsigned *bsum, long long nb) {
    __shared__ long long s_c[32];
    __shared__ long long s_tot;
    long long b, e;
    strip_of(nb, &b, &e);
    long long v = 0;
    for (long long t = b; t < e; ++t) v += bsum[t];
    long long o = block_excl_ll_pt(v, s_c, &s_tot);
    for (long long t = b; t < e; ++t) {
        const unsigned x = bsum[t];
        bsum[t] = (unsigned)o;
        o += x;
    }
}
// ------------------------------------------------------------ cluster kernels
// sort key: (shot relative to the call's first shot) << 24 | corrected ToF + bias;
// beside it each hit's pixel and ToT in one word, and the tiles' histograms of
// the first digit
template <class K>
__global__ void __launch_bounds__(GT) k_make_keys(tpx_hits h, long long n, const unsigned long long *shot_min, K *keys,
                                                  unsigned *pxt, unsigned *hist) {
    __shared__ unsigned s_h[256];
    s_h[threadIdx.x] = 0;
    const unsigned long long m = *shot_min;
    const long long base = blockIdx.x * (long long)GTILE + threadIdx.x;
    __syncthreads();
#pragma unroll
    for (int j0 = 0; j0 < GK; j0 += 4) {
        K key[4];
        unsigned px[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long i = base + (j0 + j) * GT;
            if (i >= n) continue;
            key[j] = (K)((((unsigned long long)h.shot[i] - m) << 24) | (unsigned long long)(h.tof[i] + kBias));
            px[j] = (unsigned)h.x[i] | ((unsigned)h.y[i] << 8) | ((unsigned)h.tot[i] << 16);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long i = base + (j0 + j) * GT;
            if (i >= n) continue;
            keys[i] = key[j];
            pxt[i] = px[j];
            atomicAdd(&s_h[(unsigned)key[j] & 255u], 1u);
        }
    }
    __syncthreads();
    hist[blockIdx.x * 256ll + threadIdx.x] = s_h[threadIdx.x];
}
__global__ void __launch_bounds__(GT) k_shot_range(tpx_hits h, long long n, unsigned long long *mn, unsigned long long *mx) {
    __shared__ unsigned long long s_lo[GW], s_hi[GW];
    unsigned long long lo = ~0ull, hi = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long v = (unsigned long long)h.shot[i];
        lo = min(lo, v);
        hi = max(hi, v);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_down_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_down_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        s_lo[threadIdx.x >> 5] = lo;
        s_hi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {   // one atomic pair per block: they all meet on two addresses
        for (int k = 1; k < GW; ++k) {
            lo = min(lo, s_lo[k]);
            hi = max(hi, s_hi[k]);
        }
        atomicMin(mn, lo);
        atomicMax(mx, hi);
    }
}

// the hits in sorted order, read through the sorted keys and values: shots are
// relative to the call's first one
struct Sorted {
    const unsigned *hit;            // sorted position -> hit index
    const unsigned *k32;            // the sorted keys, 32 or 64 bits wide
    const unsigned long long *k64;
    unsigned *pxt;                  // x | y << 8 | ToT << 16 in sorted order
    const int64_t *hindex;          // per hit: its stream index
    const unsigned long long *shot_min;
    __device__ __forceinline__ unsigned long long key(long long i) const { return k32 ? (unsigned long long)k32[i] : k64[i]; }
    __device__ __forceinline__ long long shot(long long i) const { return (long long)(key(i) >> 24); }
    __device__ __forceinline__ int tofb(long long i) const { return (int)(key(i) & 0xFFFFFFull); }
    __device__ __forceinline__ int x(long long i) const { return (int)(pxt[i] & 255u); }
    __device__ __forceinline__ int y(long long i) const { return (int)((pxt[i] >> 8) & 255u); }
    __device__ __forceinline__ int tot(long long i) const { return (int)(pxt[i] >> 16); }
    __device__ __forceinline__ long long index(long long i) const { return hindex[hit[i]]; }
    __device__ __forceinline__ bool emits(long long i, long long limit) const { return shot(i) + (long long)*shot_min < limit; }
};

// Counting without scan launches: a kernel counts per block of GTILE items, the
// next one adds up the counts of the blocks before its own (up to kResum
// blocks: a few loads per thread; beyond that k_scan_bsum has made the counts
// into prefixes).
constexpr long long kResum = 4096;
__device__ long long blocks_before(const unsigned *bcnt, long long nb, long long *s_w, long long *s_tot) {
    if (nb > kResum) return bcnt[blockIdx.x];
    long long v = 0;
    for (long long k = threadIdx.x; k < blockIdx.x; k += GT) v += bcnt[k];
    (void)block_scan_ll(v, s_w, s_tot);
    return *s_tot;
}
// Segments: in sorted order a gap larger than dt (or a new shot) separates
// everything before it from everything after it -- no adjacent pair spans
// it -- so each run between such gaps clusters on its own.
__device__ __forceinline__ bool seg_begins(const Sorted &s, long long i, int dt) {
    if (i == 0) return true;
    const unsigned long long a = s.key(i - 1), b = s.key(i);
    return (a >> 24) != (b >> 24) || (long long)((b & 0xFFFFFFull) - (a & 0xFFFFFFull)) > dt;
}
// counts the segments per block, and brings the pixels into sorted order
__global__ void __launch_bounds__(GT) k_seg_count(Sorted s, const unsigned *pxt_hit, long long n, int dt, unsigned *bcnt) {
    __shared__ unsigned s_c[GW];
    unsigned m[GK], total;
    const long long base = blockIdx.x * (long long)GTILE + (threadIdx.x >> 5) * (32 * GK) + (threadIdx.x & 31);
    unsigned k[GK];
#pragma unroll
    for (int j = 0; j < GK; ++j) k[j] = base + 32 * j < n ? s.hit[base + 32 * j] : 0u;
#pragma unroll
    for (int j = 0; j < GK; ++j) k[j] = pxt_hit[k[j]];
#pragma unroll
    for (int j = 0; j < GK; ++j)
        if (base + 32 * j < n) s.pxt[base + 32 * j] = k[j];
    (void)block_flags(n, [&](long long i, int) { return seg_begins(s, i, dt); }, m, s_c, &total);
    if (threadIdx.x == 0) bcnt[blockIdx.x] = total;
}
__global__ void __launch_bounds__(GT) k_seg_starts(Sorted s, long long n, int dt, const unsigned *bcnt, long long nb,
                                                   long long *start, long long *nseg) {
    __shared__ unsigned s_c[GW];
    __shared__ long long s_w[GW];
    __shared__ long long s_tot;
    unsigned m[GK], total;
    unsigned o = block_flags(n, [&](long long i, int) { return seg_begins(s, i, dt); }, m, s_c, &total);
    const long long first = blocks_before(bcnt, nb, s_w, &s_tot);
    const int lane = threadIdx.x & 31;
    const long long base = blockIdx.x * (long long)GTILE + (threadIdx.x >> 5) * (32 * GK) + lane;
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        if ((m[j] >> lane) & 1u) start[first + o + __popc(m[j] & ((1u << lane) - 1u))] = base + 32 * j;
        o += __popc(m[j]);
    }
    if (blockIdx.x == nb - 1 && threadIdx.x == 0) {
        start[first + total] = n;
        *nseg = first + total;
    }
}

// per-root moments, indexed by the hit position of the root
struct AccH { long long s_tot, s_x, s_y, s_t; unsigned n, npk; };

constexpr int WREG = 64;            // hits of a segment held in registers (two per lane)
constexpr int WCAP = 256;           // hits of a segment held by one block in shared memory
constexpr int ECAP = 1024;          // adjacent pairs of a segment kept for the hooking rounds
constexpr int HBW = 512;            // cell-hash buckets of a block's segment
constexpr int SEGW = 4;             // warps per block
struct SmallSm {                    // a segment of up to WREG hits
    int tofb[WREG];
    unsigned short tot[WREG];
    unsigned rows[16];              // occupied cells of each row of the grid
    __align__(16) unsigned short charge[256];   // ToT + 1 of a cell's hit
    __align__(8) unsigned char cell[256];
};
struct SegSm {
    int tofb[WCAP];
    int parent[WCAP];
    unsigned edge[ECAP];            // (k << 16) | j, k < j; later the roots' sums
    __align__(8) unsigned hhead[HBW];   // cell hash: first position, 0xFFFF = none; later the roots' time sums
    unsigned ecnt;
    unsigned short hnext[WCAP];
    unsigned short tot[WCAP];
    unsigned char x[WCAP], y[WCAP], np[WCAP];
};
__device__ __forceinline__ unsigned wcell(int x, int y) { return (unsigned)(x * 67 + y * 131) & (HBW - 1); }

__device__ __forceinline__ int s_find(volatile int *par, int x) {
    for (;;) {
        const int p = par[x];
        if (p == x) return x;
        const int g = par[p];
        if (g == p) return p;
        par[x] = g;
        x = g;
    }
}
// lock-free union in shared memory; the smaller position becomes the root
__device__ __forceinline__ void s_unite(int *par, int a, int b) {
    for (;;) {
        a = s_find(par, a);
        b = s_find(par, b);
        if (a == b) return;
        if (a > b) { const int t = a; a = b; b = t; }
        const int old = atomicCAS(&par[b], b, a);
        if (old == b) return;
        b = old;
    }
}

// Sec. V.B tie rule: equal ToT goes to the hit later in the stream
__device__ __forceinline__ bool j_brighter(int tj, int ti, const Sorted &s, long long j, long long i) {
    return tj > ti || (tj == ti && s.index(j) > s.index(i));
}

// Segments of at most 64 hits, in registers: lane l holds hits l and l + 32.
// For every hit k (warp-uniform loop) the ballots of "adjacent to k" give
// its adjacency row as a 64-bit mask and "brighter than k" its local-maximum
// flag; components are breadth-first closures over the rows, seeded at the
// lowest unvisited position, so the seed is the component's earliest hit.
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
struct SegIn {                      // a segment's hits in registers: two per lane
    int ta, tb;                     // ToF + bias
    unsigned a, b, ha, hb;          // pixel and ToT, hit index
    __device__ __forceinline__ void load(const Sorted &s, long long s0, long long len, int lane) {
        ta = tb = 0;
        a = b = ha = hb = 0;
        if (len > WREG) return;
        if (lane < len) { ta = s.tofb(s0 + lane); a = s.pxt[s0 + lane]; ha = s.hit[s0 + lane]; }
        if (lane + 32 < len) { tb = s.tofb(s0 + lane + 32); b = s.pxt[s0 + lane + 32]; hb = s.hit[s0 + lane + 32]; }
    }
};
__device__ __forceinline__ void seg_small(const Sorted &s, const SegIn &in, long long s0, int L, int rx, int ry, int dt, int cc, bool emit,
                          long long *labels, unsigned char *is_peak, unsigned char *rflag, AccH *acc, int lane,
                          SmallSm &W) {
    constexpr unsigned FULL = 0xffffffffu;
    const int a = lane, b = lane + 32;
    const bool va = a < L, vb = b < L;
    const int ta = in.ta, tb = in.tb;
    const unsigned pa = in.a & 0xFFFFu, pb = in.b & 0xFFFFu, oa = in.a >> 16, ob = in.b >> 16, ha = in.ha, hb = in.hb;
    unsigned long long rowA = 0, rowB = 0;
    bool npA = false, npB = false;
    // A compact segment (one particle, or a few close ones) with the 8-neighbour
    // box: its hits go into a 16 x 16 occupancy grid of their bounding box and
    // every lane reads its hits' 8 neighbour cells -- a few dozen instructions
    // per hit instead of one warp-wide step per hit of the segment. Two hits on
    // one pixel, a larger box or other radii take the all-pairs steps below.
    bool grid = false;
    // A grid segment whose hits all lie within dt of each other -- a single
    // particle, nearly always -- needs no times: local maxima from the cells'
    // charges, components by flooding rows of bits (lane r holds row r). The
    // general grid steps took 937 warp instructions per segment.
    bool flood = false;
    unsigned occ = 0;
    int ca = 0, cb = 0;             // the hits' cells
    if (rx == 1 && ry == 1) {
        const unsigned xa = pa & 255u, ya = pa >> 8, xb = pb & 255u, yb = pb >> 8;
        const unsigned x0 = __reduce_min_sync(FULL, min(va ? xa : 255u, vb ? xb : 255u));
        const unsigned x1 = __reduce_max_sync(FULL, max(va ? xa : 0u, vb ? xb : 0u));
        const unsigned y0 = __reduce_min_sync(FULL, min(va ? ya : 255u, vb ? yb : 255u));
        const unsigned y1 = __reduce_max_sync(FULL, max(va ? ya : 0u, vb ? yb : 0u));
        if (x1 - x0 <= 13u && y1 - y0 <= 13u) {
            const int t_last = __shfl_sync(FULL, L > 32 ? tb : ta, (L - 1) & 31);
            flood = t_last - __shfl_sync(FULL, ta, 0) <= dt;   // in ToF order
            unsigned char *cell = W.cell;   // 256 cells: hit + 1, 0 = empty
            __syncwarp();                   // the warp's previous segment is done with W
            reinterpret_cast<uint2 *>(cell)[lane] = make_uint2(0u, 0u);
            reinterpret_cast<uint4 *>(W.charge)[lane] = make_uint4(0u, 0u, 0u, 0u);
            if (lane < 16) W.rows[lane] = 0u;
            if (va) { W.tofb[a] = ta; W.tot[a] = (unsigned short)oa; }
            if (vb) { W.tofb[b] = tb; W.tot[b] = (unsigned short)ob; }
            __syncwarp();
            ca = (int)(xa - x0 + 1) + 16 * (int)(ya - y0 + 1);
            cb = (int)(xb - x0 + 1) + 16 * (int)(yb - y0 + 1);
            if (va) { cell[ca] = (unsigned char)(a + 1); W.charge[ca] = (unsigned short)(oa + 1u); atomicOr(&W.rows[ca >> 4], 1u << (ca & 15)); }
            if (vb) { cell[cb] = (unsigned char)(b + 1); W.charge[cb] = (unsigned short)(ob + 1u); atomicOr(&W.rows[cb >> 4], 1u << (cb & 15)); }
            __syncwarp();
            // a hit that does not find itself shares its pixel with another
            grid = !__any_sync(FULL, (va && cell[ca] != a + 1) || (vb && cell[cb] != b + 1));
            flood = flood && grid && oa < 65535u && ob < 65535u;
            flood = __all_sync(FULL, flood);
            if (flood) {
                occ = lane < 16 ? W.rows[lane] : 0u;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!(h ? vb : va)) continue;
                    const int c = h ? cb : ca;
                    const unsigned o1 = (h ? ob : oa) + 1u;
                    unsigned mx = 0;
#pragma unroll
                    for (int d = 0; d < 9; ++d)
                        if (d != 4) mx = max(mx, (unsigned)W.charge[c + (d % 3 - 1) + 16 * (d / 3 - 1)]);
                    bool np = mx > o1;
                    if (mx == o1) {   // Sec. V.B ties: the later hit in the stream wins
                        for (int d = 0; d < 9; ++d) {
                            const int cj = c + (d % 3 - 1) + 16 * (d / 3 - 1);
                            if (d != 4 && W.charge[cj] == o1 && s.index(s0 + cell[cj] - 1) > (long long)s.hindex[h ? hb : ha]) np = true;
                        }
                    }
                    if (h) npB = np; else npA = np;
                }
            }
            if (grid && !flood) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool v = h ? vb : va;
                    if (!v) continue;
                    const int c = h ? cb : ca, t = h ? tb : ta;
                    const unsigned o = h ? ob : oa;
                    unsigned long long row = 0;
                    bool np = false;
#pragma unroll
                    for (int d = 0; d < 9; ++d) {
                        if (d == 4) continue;
                        const unsigned j1 = cell[c + (d % 3 - 1) + 16 * (d / 3 - 1)];
                        if (!j1) continue;
                        const int j = (int)j1 - 1;
                        if (abs(W.tofb[j] - t) > dt) continue;
                        row |= 1ull << j;
                        const unsigned oj = W.tot[j];
                        if (oj > o || (oj == o && s.index(s0 + j) > (long long)s.hindex[h ? hb : ha])) np = true;
                    }
                    if (h) { rowB = row; npB = np; } else { rowA = row; npA = np; }
                }
            }
            __syncwarp();
        }
    }
    const unsigned rxy = (unsigned)rx | ((unsigned)ry << 8);   // per-byte box radii
    for (int k = 0; k < (grid ? 0 : L); ++k) {
        const bool kb = k >= 32;
        const int src = k & 31;
        const int kt = __shfl_sync(FULL, kb ? tb : ta, src);
        const unsigned kp = __shfl_sync(FULL, kb ? pb : pa, src);
        const unsigned ko = __shfl_sync(FULL, kb ? ob : oa, src);
        const bool adjA = va && a != k && abs(ta - kt) <= dt && __vcmpleu4(__vabsdiffu4(pa, kp), rxy) == FULL;
        const bool adjB = vb && b != k && abs(tb - kt) <= dt && __vcmpleu4(__vabsdiffu4(pb, kp), rxy) == FULL;
        const unsigned lo = __ballot_sync(FULL, adjA), hi = __ballot_sync(FULL, adjB);
        bool brA = adjA && oa > ko, brB = adjB && ob > ko;
        const bool tA = adjA && oa == ko, tB = adjB && ob == ko;
        if (__any_sync(FULL, tA || tB)) {   // Sec. V.B ties: the later hit in the stream wins
            const long long ki = s.index(s0 + k);
            brA = brA || (tA && (long long)s.hindex[ha] > ki);
            brB = brB || (tB && (long long)s.hindex[hb] > ki);
        }
        const bool knp = __any_sync(FULL, brA || brB);
        if (lane == src) {
            const unsigned long long row = ((unsigned long long)hi << 32) | lo;
            if (kb) { rowB = row; npB = knp; } else { rowA = row; npA = knp; }
        }
    }
    const bool pkA = va && !npA, pkB = vb && !npB;
    if (!cc) {   // PAPER mode: every hit is its own label; local maxima carry the records
        if (va) {
            if (labels) labels[ha] = s.hindex[ha];
            if (is_peak) is_peak[ha] = pkA;
            if (rflag) rflag[ha] = emit && pkA;
        }
        if (vb) {
            if (labels) labels[hb] = s.hindex[hb];
            if (is_peak) is_peak[hb] = pkB;
            if (rflag) rflag[hb] = emit && pkB;
        }
        return;
    }
    // the hits' stream indices, for the labels: on their way during the closures
    const long long ia = labels && va ? (long long)s.hindex[ha] : 0, ib = labels && vb ? (long long)s.hindex[hb] : 0;
    const unsigned long long peaks = ((unsigned long long)__ballot_sync(FULL, pkB) << 32) | __ballot_sync(FULL, pkA);
    unsigned long long todo = L == 64 ? ~0ull : ((1ull << L) - 1ull);
    long long rootA = 0, rootB = 0;
    int rposA = -1, rposB = -1;
    while (todo) {
        const int seed = __ffsll((long long)todo) - 1;
        unsigned long long comp = 1ull << seed, front = comp;
        if (flood) {
            const int sc = __shfl_sync(FULL, seed >= 32 ? cb : ca, seed & 31);
            unsigned f = lane == (sc >> 4) ? 1u << (sc & 15) : 0u;
            for (;;) {
                const unsigned was = f;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const unsigned e = f | (f << 1) | (f >> 1);
                    f = (e | __shfl_up_sync(FULL, e, 1) | __shfl_down_sync(FULL, e, 1)) & occ;
                }
                if (!__any_sync(FULL, f != was)) break;
            }
            const unsigned fa = __shfl_sync(FULL, f, ca >> 4), fb = __shfl_sync(FULL, f, cb >> 4);
            const unsigned lo = __ballot_sync(FULL, va && ((fa >> (ca & 15)) & 1u));
            const unsigned hi = __ballot_sync(FULL, vb && ((fb >> (cb & 15)) & 1u));
            comp = ((unsigned long long)hi << 32) | lo;
            front = 0;
        }
        while (front) {
            unsigned long long c = 0;
            if ((front >> a) & 1ull) c |= rowA;
            if ((front >> b) & 1ull) c |= rowB;
            const unsigned lo = __reduce_or_sync(FULL, (unsigned)c);
            const unsigned hi = __reduce_or_sync(FULL, (unsigned)(c >> 32));
            const unsigned long long nb = ((unsigned long long)hi << 32) | lo;
            front = nb & ~comp;
            comp |= nb;
        }
        const long long sidx = labels ? __shfl_sync(FULL, seed >= 32 ? ib : ia, seed & 31) : 0;
        const bool inA = (comp >> a) & 1ull, inB = (comp >> b) & 1ull;
        if (inA) { rootA = sidx; rposA = seed; }
        if (inB) { rootB = sidx; rposB = seed; }
        if (acc && emit) {
            const int st = __shfl_sync(FULL, seed >= 32 ? tb : ta, seed & 31);
            // 64 hits: ToT sums and their products with a coordinate fit 32 bits
            unsigned v_tot = 0, v_x = 0, v_y = 0;
            unsigned long long v_t = 0;
            if (inA) { v_tot += oa; v_x += oa * (pa & 255u); v_y += oa * (pa >> 8); v_t += (unsigned long long)(ta - st) * oa; }
            if (inB) { v_tot += ob; v_x += ob * (pb & 255u); v_y += ob * (pb >> 8); v_t += (unsigned long long)(tb - st) * ob; }
            v_tot = __reduce_add_sync(FULL, v_tot);
            v_x = __reduce_add_sync(FULL, v_x);
            v_y = __reduce_add_sync(FULL, v_y);
            // 64 hits within 63 dt of each other: also s_t for dt <= 1000 and 10-bit ToT
            if (dt <= 1000 && __all_sync(FULL, (oa | ob) < 1024u)) v_t = __reduce_add_sync(FULL, (unsigned)v_t);
            else v_t = warp_sum_u64(v_t);
            if (lane == (seed & 31)) {
                AccH r;
                r.s_tot = v_tot; r.s_x = v_x; r.s_y = v_y; r.s_t = (long long)v_t;
                r.n = (unsigned)__popcll(comp); r.npk = (unsigned)__popcll(comp & peaks);
                acc[seed >= 32 ? hb : ha] = r;
            }
        }
        todo &= ~comp;
    }
    if (va) {
        if (labels) labels[ha] = rootA;
        if (is_peak) is_peak[ha] = pkA;
        if (rflag) rflag[ha] = emit && rposA == a;
    }
    if (vb) {
        if (labels) labels[hb] = rootB;
        if (is_peak) is_peak[hb] = pkB;
        if (rflag) rflag[hb] = emit && rposB == b;
    }
}

// One warp per segment of up to 64 hits, in registers (seg_small) and 1,300
// bytes of shared memory; the rare longer segments are listed for
// k_segments_mid (up to WCAP) or marked for the cell-hash kernels in global
// memory below. Bound by instruction issue: 6.0e6 hits 402 -> 141 us, of which
// the longer segments' 11 KB of shared memory taken out of this kernel 190, the
// flooding of bit rows (below) 85.
struct SegLists { unsigned n_mid, n_long; };
__global__ void __launch_bounds__(SEGW * 32, 8) k_segments(Sorted s, const long long *seg_start, const long long *nseg_p,
                                                           int rx, int ry, int dt, int cc, long long shot_limit,
                                                           long long *labels, unsigned char *is_peak,
                                                           unsigned char *rflag, AccH *acc, unsigned char *mark,
                                                           unsigned *mid, SegLists *lists) {
    __shared__ SmallSm sm[SEGW];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const long long nseg = *nseg_p;
    for (long long seg = blockIdx.x * (long long)SEGW + wi; seg < nseg; seg += (long long)gridDim.x * SEGW) {
        const long long s0 = seg_start[seg], len = seg_start[seg + 1] - s0;
        SegIn in;
        in.load(s, s0, len, lane);
        for (long long k = lane; k < len; k += 32) mark[s0 + k] = len > WCAP;
        if (len > WREG) {
            if (lane == 0) {
                if (len > WCAP) lists->n_long = 1;
                else mid[atomicAdd(&lists->n_mid, 1u)] = (unsigned)seg;
            }
        } else {
            const bool emit = s.emits(s0, shot_limit);
            const bool sums = cc && acc && emit;
            if (len > 1) {
                seg_small(s, in, s0, (int)len, rx, ry, dt, cc, emit, labels, is_peak, rflag, sums ? acc : nullptr, lane, sm[wi]);
            } else if (lane == 0) {
                if (labels) labels[in.ha] = s.hindex[in.ha];
                if (is_peak) is_peak[in.ha] = 1;
                if (rflag) rflag[in.ha] = emit;
                if (sums) {
                    const long long t = in.a >> 16;
                    AccH v;
                    v.s_tot = t; v.s_x = t * (in.a & 255u); v.s_y = t * ((in.a >> 8) & 255u); v.s_t = 0; v.n = 1; v.npk = 1;
                    acc[in.ha] = v;
                }
            }
        }
    }
}

// Segments of 65 to WCAP hits: one block in shared memory, where a cell hash of
// the segment gives every hit the candidates of the forward half of its box
// (same cell: later positions only), so that each adjacent pair is met once
// even when the whole segment lies within dt; pairs set the local-maximum flags
// and are joined by hooking rounds; then labels, peaks, root flags (emitted
// shots only) and the root's int64 moments. Bound by the steps that follow one
// another in a segment: with a warp per segment 6.0e6 hits took 89 us,
// 4e5 hits 43; with a block 53 and 22.
__global__ void __launch_bounds__(SEGW * 32) k_segments_mid(Sorted s, const long long *seg_start, const unsigned *mid,
                                                            const SegLists *lists, int rx, int ry, int dt, int cc,
                                                            long long shot_limit, long long *labels,
                                                            unsigned char *is_peak, unsigned char *rflag, AccH *acc) {
    __shared__ SegSm W;
    const int lane = threadIdx.x & 31, tid = threadIdx.x;
    constexpr int TH = SEGW * 32;
    const long long n_mid = lists->n_mid;
    for (long long q = blockIdx.x; q < n_mid; q += gridDim.x) {
        const long long s0 = seg_start[mid[q]];
        const int L = (int)(seg_start[mid[q] + 1ll] - s0);
        const bool emit = s.emits(s0, shot_limit);
        const bool sums = cc && acc && emit;
        for (int k = tid; k < L; k += TH) {
            W.tofb[k] = s.tofb(s0 + k);
            W.x[k] = s.x(s0 + k);
            W.y[k] = s.y(s0 + k);
            W.tot[k] = s.tot(s0 + k);
            W.parent[k] = k;
            W.np[k] = 0;
        }
        for (int b = tid; b < HBW; b += TH) W.hhead[b] = 0xFFFFu;
        if (tid == 0) W.ecnt = 0;
        __syncthreads();
        for (int k = tid; k < L; k += TH) W.hnext[k] = (unsigned short)atomicExch(&W.hhead[wcell(W.x[k], W.y[k])], (unsigned)k);
        __syncthreads();
        for (int k = tid; k < L; k += TH) {
            const int tb = W.tofb[k], xk = W.x[k], yk = W.y[k], tk = W.tot[k];
            for (int dx = 0; dx <= rx; ++dx) {
                const int cx = xk + dx;
                if (cx > 255) break;
                for (int dy = (dx == 0 ? 0 : -ry); dy <= ry; ++dy) {
                    const int cy = yk + dy;
                    if (cy < 0 || cy > 255) continue;
                    for (unsigned j = W.hhead[wcell(cx, cy)]; j != 0xFFFFu; j = W.hnext[j]) {
                        if (dx == 0 && dy == 0 && (int)j <= k) continue;
                        if (W.x[j] != cx || W.y[j] != cy) continue;
                        const int d = W.tofb[j] - tb;
                        if (d < -dt || d > dt) continue;
                        // the pair (lo, hi) in position order
                        const int lo = min(k, (int)j), hi = max(k, (int)j);
                        if (j_brighter(W.tot[j], tk, s, s0 + j, s0 + k)) W.np[k] = 1; else W.np[j] = 1;
                        if (cc) {   // record the pair (warp-aggregated slot); beyond the buffer, join it now
                            const unsigned am = __activemask();
                            const int leader = __ffs(am) - 1;
                            unsigned slot = 0;
                            if (lane == leader) slot = atomicAdd(&W.ecnt, (unsigned)__popc(am));
                            slot = __shfl_sync(am, slot, leader) + __popc(am & ((1u << lane) - 1u));
                            if (slot < (unsigned)ECAP) W.edge[slot] = ((unsigned)lo << 16) | (unsigned)hi;
                            else s_unite(W.parent, lo, hi);
                        }
                    }
                }
            }
        }
        __syncthreads();
        if (cc) {
            // rounds of: pointer jumping until every hit points at its root,
            // then every recorded pair whose roots differ hooks the larger
            // root onto the smaller one (CAS on a root only, so no link is
            // ever overwritten); until no pair has two roots. Pointers only
            // go to smaller positions, so the root is the earliest hit.
            const int m = min((int)W.ecnt, ECAP);
            for (;;) {
                for (;;) {
                    bool moved = false;
                    for (int k = tid; k < L; k += TH) {
                        const int p = W.parent[k], pp = W.parent[p];
                        if (pp != p) { W.parent[k] = pp; moved = true; }
                    }
                    if (!__syncthreads_or(moved)) break;
                }
                bool hooked = false;
                for (int e = tid; e < m; e += TH) {
                    const unsigned ed = W.edge[e];
                    const int a = W.parent[ed >> 16], b = W.parent[ed & 0xFFFFu];
                    if (a != b) {
                        atomicCAS(&W.parent[max(a, b)], max(a, b), min(a, b));
                        hooked = true;
                    }
                }
                if (!__syncthreads_or(hooked)) break;
            }
        }
        __syncthreads();
        // roots of every hit (full compression; only reads after the barrier)
        int rk[WCAP / TH];
#pragma unroll
        for (int u = 0; u < WCAP / TH; ++u) {
            const int k = u * TH + tid;
            rk[u] = (k < L && cc) ? s_find(W.parent, k) : k;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < WCAP / TH; ++u) {
            const int k = u * TH + tid;
            if (k < L) W.parent[k] = rk[u];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < WCAP / TH; ++u) {
            const int k = u * TH + tid;
            if (k >= L) break;
            const int r = rk[u];
            const unsigned hh = s.hit[s0 + k];
            const bool peak = W.np[k] == 0;
            if (labels) labels[hh] = s.index(s0 + r);
            if (is_peak) is_peak[hh] = peak;
            if (rflag) rflag[hh] = emit && (cc ? r == k : peak);
        }
        if (sums) {
            // every hit adds to its root's sums in the space of the pair list and
            // the hash heads: 256 hits, so ToT sums times a coordinate fit 32 bits
            unsigned *q_n = W.edge, *q_tot = q_n + WCAP, *q_x = q_tot + WCAP, *q_y = q_x + WCAP;
            unsigned long long *q_t = reinterpret_cast<unsigned long long *>(W.hhead);
            for (int k = tid; k < L; k += TH) {
                q_n[k] = q_tot[k] = q_x[k] = q_y[k] = 0u;
                q_t[k] = 0ull;
            }
            __syncthreads();
            for (int k = tid; k < L; k += TH) {
                const int r = W.parent[k];
                const unsigned t = W.tot[k];
                atomicAdd(&q_n[r], 1u | (W.np[k] == 0 ? 1u << 16 : 0u));
                atomicAdd(&q_tot[r], t);
                atomicAdd(&q_x[r], t * W.x[k]);
                atomicAdd(&q_y[r], t * W.y[k]);
                atomicAdd(&q_t[r], (unsigned long long)(W.tofb[k] - W.tofb[r]) * t);
            }
            __syncthreads();
            for (int k = tid; k < L; k += TH) {
                if (W.parent[k] != k) continue;
                AccH a;
                a.s_tot = q_tot[k]; a.s_x = q_x[k]; a.s_y = q_y[k]; a.s_t = (long long)q_t[k];
                a.n = q_n[k] & 0xFFFFu; a.npk = q_n[k] >> 16;
                acc[s.hit[s0 + k]] = a;
            }
        }
        __syncthreads();
    }
}

// ---- segments longer than WCAP: the same rules through global memory ----
__device__ __forceinline__ int g_find(int *parent, int x) {
    for (;;) {
        const int p = ((volatile int *)parent)[x];
        if (p == x) return x;
        const int g = ((volatile int *)parent)[p];
        if (g == p) return p;
        ((volatile int *)parent)[x] = g;
        x = g;
    }
}
__device__ void g_unite(int *parent, int a, int b) {
    for (;;) {
        a = g_find(parent, a);
        b = g_find(parent, b);
        if (a == b) return;
        if (a > b) { const int t = a; a = b; b = t; }
        const int old = atomicCAS(&parent[b], b, a);
        if (old == b) return;
        b = old;
    }
}
// (every k_long_ kernel returns at once when no segment is that long)
__global__ void k_long_init(Sorted s, long long n, const SegLists *lists, const unsigned char *mark, int *parent,
                            unsigned char *notpeak, AccH *acc, unsigned *head, unsigned long long mask) {
    if (!lists->n_long) return;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i <= mask; i += (unsigned long long)gridDim.x * blockDim.x)
        head[i] = 0xFFFFFFFFu;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (!mark[i]) continue;
        parent[i] = (int)i;
        notpeak[i] = 0;
        if (acc) {
            AccH z;
            z.s_tot = 0; z.s_x = 0; z.s_y = 0; z.s_t = 0; z.n = 0; z.npk = 0;
            acc[s.hit[i]] = z;
        }
    }
}
// Long segments can hold thousands of hits within dt of each other (a shot
// of many particles arriving together), so their pairs come from a hash of
// (shot, x, y) cells: every hit looks up the cells of the forward half of its
// box (same cell: later positions only), which meets each adjacent pair once.
__device__ __forceinline__ unsigned long long cell_hash(long long shot, int x, int y, unsigned long long mask) {
    unsigned long long k = ((unsigned long long)shot << 16) ^ ((unsigned long long)x << 8) ^ (unsigned long long)y;
    k *= 0x9E3779B97F4A7C15ull;   // Fibonacci hashing
    return (k >> 20) & mask;
}
// a marked hit's cell and time in one word for the pair search: x, y, the
// shot's low 16 bits, ToF + bias (the full shot is compared on a match)
__device__ __forceinline__ unsigned cell_key(long long shot, int x, int y) {
    return (unsigned)x | ((unsigned)y << 8) | ((unsigned)(shot & 0xFFFF) << 16);
}
__global__ void k_long_insert(Sorted s, long long n, const SegLists *lists, const unsigned char *mark, unsigned *head,
                              unsigned *next, unsigned long long *word, unsigned long long mask) {
    if (!lists->n_long) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (!mark[i]) continue;
        const long long sh = s.shot(i);
        const int x = s.x(i), y = s.y(i);
        word[i] = (unsigned long long)cell_key(sh, x, y) | ((unsigned long long)(unsigned)s.tofb(i) << 32);
        next[i] = atomicExch(&head[cell_hash(sh, x, y, mask)], (unsigned)i);
    }
}
__global__ void k_long_pairs(Sorted s, long long n, const SegLists *lists, const unsigned char *mark,
                             const unsigned *head, const unsigned *next, const unsigned long long *word,
                             unsigned long long mask, int rx, int ry, int dt, int cc, int *parent,
                             unsigned char *notpeak) {
    if (!lists->n_long) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (!mark[i]) continue;
        const unsigned long long wi = word[i];
        const long long sh = s.shot(i);
        const int tb = (int)(unsigned)(wi >> 32), xi = (int)(wi & 255), yi = (int)((wi >> 8) & 255), ti = s.tot(i);
        for (int dx = 0; dx <= rx; ++dx) {
            const int cx = xi + dx;
            if (cx > 255) break;
            for (int dy = (dx == 0 ? 0 : -ry); dy <= ry; ++dy) {
                const int cy = yi + dy;
                if (cy < 0 || cy > 255) continue;
                const unsigned key = cell_key(sh, cx, cy);
                for (unsigned j = head[cell_hash(sh, cx, cy, mask)]; j != 0xFFFFFFFFu; j = next[j]) {
                    if (dx == 0 && dy == 0 && (long long)j <= i) continue;
                    const unsigned long long wj = word[j];
                    if ((unsigned)wj != key || s.shot(j) != sh) continue;
                    const int d = (int)(unsigned)(wj >> 32) - tb;
                    if (d < -dt || d > dt) continue;
                    if (j_brighter(s.tot(j), ti, s, j, i)) notpeak[i] = 1; else notpeak[j] = 1;
                    if (cc) g_unite(parent, (int)i, (int)j);
                }
            }
        }
    }
}
__global__ void k_long_finish(Sorted s, long long n, const SegLists *lists, const unsigned char *mark, int cc,
                              long long shot_limit, int *parent, const unsigned char *notpeak, long long *labels,
                              unsigned char *is_peak, unsigned char *rflag, AccH *acc) {
    if (!lists->n_long) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (!mark[i]) continue;
        const long long r = cc ? g_find(parent, (int)i) : i;
        const unsigned hh = s.hit[i];
        const bool peak = notpeak[i] == 0, emit = s.emits(i, shot_limit);
        if (labels) labels[hh] = s.index(r);
        if (is_peak) is_peak[hh] = peak;
        if (rflag) rflag[hh] = emit && (cc ? r == i : peak);
        if (cc && acc && emit) {
            AccH &a = acc[s.hit[r]];
            const unsigned long long t = s.tot(i);
            atomicAdd(reinterpret_cast<unsigned long long *>(&a.s_tot), t);
            atomicAdd(reinterpret_cast<unsigned long long *>(&a.s_x), t * s.x(i));
            atomicAdd(reinterpret_cast<unsigned long long *>(&a.s_y), t * s.y(i));
            atomicAdd(reinterpret_cast<unsigned long long *>(&a.s_t), (unsigned long long)(s.tofb(i) - s.tofb(r)) * t);
            atomicAdd(&a.n, 1u);
            if (peak) atomicAdd(&a.npk, 1u);
        }
    }
}

// ------------------------------------------------------------ centroid kernels
// Records in ascending label order: the roots (CC mode: the hits that carry
// their own label; PAPER mode: the local maxima) are counted per block of
// GTILE hits, then every block places its own behind those of the blocks
// before it.
struct RootFlag {
    const long long *labels, *index;    // CC mode from labels
    const unsigned char *flag;          // or flags as they are
    __device__ __forceinline__ bool operator()(long long i, int) const { return flag ? flag[i] != 0 : labels[i] == index[i]; }
};
__global__ void __launch_bounds__(GT) k_root_count(RootFlag f, long long n, unsigned *bcnt) {
    __shared__ unsigned s_c[GW];
    unsigned m[GK], total;
    (void)block_flags(n, f, m, s_c, &total);
    if (threadIdx.x == 0) bcnt[blockIdx.x] = total;
}
// latches the number of records, the capacity status and the clusters counter
__device__ __forceinline__ void latch_count(long long m, long long cap, long long *n_rec, unsigned *status,
                                            unsigned long long *counter) {
    *n_rec = m;
    if (m > cap) atomicOr(status, ST_CLUSTER_CAP);
    if (counter) *counter = (unsigned long long)m;
}
__device__ __forceinline__ void write_record(const tpx_hits &h, long long i, const AccH &a, tpx_record *out) {
    tpx_record o;
    o.label = h.index[i];
    o.shot = h.shot[i];
    o.t0 = h.t[i];
    o.s_tot = a.s_tot; o.s_x = a.s_x; o.s_y = a.s_y; o.s_t = a.s_t;
    o.n = (int)a.n; o.n_peaks = (int)a.npk;
    com_from_moments(o.s_x, o.s_y, o.s_t, o.s_tot, h.tof[i], &o.x, &o.y, &o.tof);
    *out = o;
}
// places the roots; one of three uses: `out` (with acc, per hit): the records
// themselves; `zero`: each record's empty sums and its root, for k_accum (and
// `rank`, the record of a root's label, when the labels' span allows it); `cid`
// (per hit): the roots' slots, for k_paper
struct Roots {
    const AccH *acc; tpx_record *out;
    unsigned *cid;
    unsigned *rank; long long rank_cap;
    struct Acc *zero; unsigned *rootpos; long long *root_t;
};
struct Acc { unsigned long long n_npk, s_tot, s_x, s_y, s_t; };   // n_npk: hits | local maxima << 32
__global__ void __launch_bounds__(GT) k_root_place(RootFlag f, tpx_hits h, long long n, const unsigned *bcnt, long long nb,
                                                   long long cap, long long *n_rec, unsigned *status,
                                                   unsigned long long *counter, Roots r) {
    __shared__ unsigned s_c[GW];
    __shared__ long long s_w[GW];
    __shared__ long long s_tot;
    __shared__ unsigned s_root[GTILE];
    unsigned m[GK], total;
    unsigned o = block_flags(n, f, m, s_c, &total);
    const long long first = blocks_before(bcnt, nb, s_w, &s_tot);
    const int lane = threadIdx.x & 31;
    const int at = (threadIdx.x >> 5) * (32 * GK) + lane;
    const long long base = blockIdx.x * (long long)GTILE;
#pragma unroll
    for (int j = 0; j < GK; ++j) {
        if ((m[j] >> lane) & 1u) {
            const unsigned k = o + __popc(m[j] & ((1u << lane) - 1u));
            s_root[k] = (unsigned)(at + 32 * j);
        }
        o += __popc(m[j]);
    }
    __syncthreads();
    const bool ranked = r.rank && h.index[n - 1] - h.index[0] < r.rank_cap;
    for (unsigned k = threadIdx.x; k < total; k += GT) {
        const long long i = base + s_root[k], c = first + k;
        if (r.cid) r.cid[i] = (unsigned)c;
        if (c < cap && r.out && r.acc) write_record(h, i, r.acc[i], r.out + c);
        if (c < cap && r.zero) {
            r.zero[c] = Acc{0, 0, 0, 0, 0};
            r.rootpos[c] = (unsigned)i;
            r.root_t[c] = h.t[i];
            const long long at = h.index[i] - h.index[0];
            if (ranked && at >= 0 && at < r.rank_cap) r.rank[at] = (unsigned)c;
        }
    }
    if (blockIdx.x == nb - 1 && threadIdx.x == 0) latch_count(first + total, cap, n_rec, status, counter);
}

// Every hit adds to its record's sums. The record comes from the rank table
// (4 bytes per stream index; a binary search over the roots where the indices
// span more). A block's 4096 hits in stream order belong to a few hundred
// records, so they meet in a hash table in shared memory first, in 32 bits
// (4096 hits: ToT sums times a coordinate fit; s_t for times within 1023 ticks
// of the root, else past the table), and its entries go to global memory.
// With six 64-bit global atomics and a 23-step search per hit, 6.0e6 hits
// took 264 us; 92 with one hit's loads in flight per thread, 71 with four's.
constexpr int AH = 1024;            // hash slots: a quarter of a block's hits
__global__ void __launch_bounds__(GT) k_accum(tpx_hits h, const long long *labels, const unsigned char *is_peak, long long n,
                                              const long long *n_rec, long long cap, const unsigned *rank,
                                              long long rank_cap, const unsigned *rootpos, const long long *root_t,
                                              Acc *acc) {
    __shared__ unsigned s_key[AH];      // record + 1, 0: free
    __shared__ unsigned s_n[AH], s_p[AH], s_t[AH], s_x[AH], s_y[AH], s_d[AH];
    for (int k = threadIdx.x; k < AH; k += GT) s_key[k] = s_n[k] = s_p[k] = s_t[k] = s_x[k] = s_y[k] = s_d[k] = 0u;
    __syncthreads();
    const long long m = min(*n_rec, cap);
    const long long i0 = h.index[0], span = h.index[n - 1] - i0;
    const bool ranked = span < rank_cap;
    const long long base = blockIdx.x * (long long)GTILE;
    constexpr int B = 4;   // hits whose loads are in flight together
    for (int j0 = 0; j0 < GK; j0 += B) {
        long long rec[B], t[B];
        unsigned xyt[B], pks[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const long long i = base + (j0 + j) * GT + threadIdx.x;
            rec[j] = -1;
            if (i >= n) continue;
            rec[j] = labels[i];
            t[j] = h.t[i];
            xyt[j] = (unsigned)h.x[i] | ((unsigned)h.y[i] << 8) | ((unsigned)h.tot[i] << 16);
            pks[j] = is_peak && is_peak[i] ? 1u : 0u;
        }
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const long long lab = rec[j];
            const bool in = base + (j0 + j) * GT + threadIdx.x < n;
            if (ranked) {   // no record's label: the table's 2^32 - 1, past every count
                rec[j] = in && lab >= i0 && lab - i0 <= span ? (long long)rank[lab - i0] : -1;
            } else {
                long long lo = 0, hi = in ? m : 0;   // the record whose root carries the label
                while (lo < hi) {
                    const long long mid = lo + ((hi - lo) >> 1);
                    if (h.index[rootpos[mid]] < lab) lo = mid + 1; else hi = mid;
                }
                rec[j] = in && lo < m && h.index[rootpos[lo]] == lab ? lo : -1;
            }
        }
#pragma unroll
        for (int j = 0; j < B; ++j)
            if (rec[j] >= 0 && rec[j] < m) t[j] -= root_t[rec[j]];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const long long c = rec[j], d = t[j];
            if (c < 0 || c >= m) continue;   // past the capacity, or no record's label
            const unsigned tot = xyt[j] >> 16, x = xyt[j] & 255u, y = (xyt[j] >> 8) & 255u, pk = pks[j];
            unsigned slot = (unsigned)c * 2654435761u >> 22;   // AH = 2^10 slots
            int probe = tot < 1024u ? 0 : 8;   // larger ones (not from packets) could overflow the table's sums
            for (; probe < 8; ++probe, slot = (slot + 1) & (AH - 1)) {
                const unsigned k = atomicCAS(&s_key[slot], 0u, (unsigned)c + 1u);
                if (k == 0u || k == (unsigned)c + 1u) break;
            }
            if (probe < 8) {
                atomicAdd(&s_n[slot], 1u);
                if (pk) atomicAdd(&s_p[slot], 1u);
                atomicAdd(&s_t[slot], tot);
                atomicAdd(&s_x[slot], tot * x);
                atomicAdd(&s_y[slot], tot * y);
                if (d >= 0 && d < 1024) atomicAdd(&s_d[slot], tot * (unsigned)d);
                else atomicAdd(&acc[c].s_t, tot * (unsigned long long)d);
            } else {
                atomicAdd(&acc[c].n_npk, 1ull | ((unsigned long long)pk << 32));
                atomicAdd(&acc[c].s_tot, (unsigned long long)tot);
                atomicAdd(&acc[c].s_x, (unsigned long long)tot * x);
                atomicAdd(&acc[c].s_y, (unsigned long long)tot * y);
                atomicAdd(&acc[c].s_t, tot * (unsigned long long)d);
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < AH; k += GT) {
        if (!s_key[k]) continue;
        Acc &a = acc[s_key[k] - 1u];
        atomicAdd(&a.n_npk, s_n[k] | ((unsigned long long)s_p[k] << 32));
        atomicAdd(&a.s_tot, (unsigned long long)s_t[k]);
        atomicAdd(&a.s_x, (unsigned long long)s_x[k]);
        atomicAdd(&a.s_y, (unsigned long long)s_y[k]);
        if (s_d[k]) atomicAdd(&a.s_t, (unsigned long long)s_d[k]);
    }
}

__global__ void k_final(tpx_hits h, const long long *n_rec, long long cap, const unsigned *rootpos, const Acc *acc,
                        tpx_record *out) {
    const long long m = min(*n_rec, cap);
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < m; c += (long long)gridDim.x * blockDim.x) {
        const Acc a = acc[c];
        AccH v;
        v.s_tot = (long long)a.s_tot; v.s_x = (long long)a.s_x; v.s_y = (long long)a.s_y; v.s_t = (long long)a.s_t;
        v.n = (unsigned)a.n_npk; v.npk = (unsigned)(a.n_npk >> 32);
        write_record(h, rootpos[c], v, out + c);
    }
}

// PAPER mode: each local maximum sums its box neighbourhood (both directions
// in sorted order, within dt)
__global__ void k_paper(Sorted s, long long n, int rx, int ry, int dt, const unsigned char *flag_hit,
                        const unsigned *cid_hit, tpx_hits h, tpx_record *out, long long cap) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned hi = s.hit[i];
        if (!flag_hit[hi]) continue;
        const long long c = cid_hit[hi];
        if (c >= cap) continue;
        const long long sh = s.shot(i);
        const int tb = s.tofb(i), xi = s.x(i), yi = s.y(i);
        long long m = 0, st = 0, sx = 0, sy = 0, a2 = 0;
        int tmin = tb;
        for (int dir = -1; dir <= 1; dir += 2) {
            for (long long j = (dir < 0 ? i : i + 1); j >= 0 && j < n; j += dir) {
                if (s.shot(j) != sh) break;
                const int d = s.tofb(j) - tb;
                if (d > dt || d < -dt) break;
                const int dx = (int)s.x(j) - xi, dy = (int)s.y(j) - yi;
                if (dx < -rx || dx > rx || dy < -ry || dy > ry) continue;
                const long long tj = s.tot(j);
                m += 1; st += tj; sx += tj * s.x(j); sy += tj * s.y(j); a2 += tj * s.tofb(j);
                tmin = min(tmin, s.tofb(j));
            }
        }
        tpx_record o;
        o.label = s.index(i);
        o.shot = h.shot[hi];
        const long long tofc0 = (long long)tmin - kBias;
        o.t0 = h.t[hi] - h.tof[hi] + tofc0;
        o.s_tot = st; o.s_x = sx; o.s_y = sy; o.s_t = a2 - (long long)tmin * st;
        o.n = (int)m; o.n_peaks = 1;
        com_from_moments(sx, sy, o.s_t, st, tofc0, &o.x, &o.y, &o.tof);
        out[c] = o;
    }
}

// ------------------------------------------------------------ host helpers
// a failed CUDA call becomes TPX_ECUDA; with TPX_DEBUG set in the
// environment its error is also printed to stderr
inline int ck(cudaError_t e, int line = __builtin_LINE()) {
    if (e == cudaSuccess) return TPX_OK;
    if (std::getenv("TPX_DEBUG")) std::fprintf(stderr, "tpx_general.cu:%d: %s\n", line, cudaGetErrorString(e));
    return TPX_ECUDA;
}
inline unsigned grid_for(long long n) {
    long long g = (n + GT - 1) / GT;
    if (g < 1) g = 1;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)g;
}

struct Arena {
    char *p;
    size_t used, cap;
    template <class T>
    T *take(long long count) {
        const size_t b = ((size_t)(count > 0 ? count : 1) * sizeof(T) + 255) & ~size_t(255);
        T *r = reinterpret_cast<T *>(p + used);
        used += b;
        return r;
    }
};
inline size_t sz(long long count, size_t elem) { return ((size_t)(count > 0 ? count : 1) * elem + 255) & ~size_t(255); }

int reserve(tpx_ctx *c, size_t bytes) {
    if (c->g_mem && c->g_bytes >= bytes) return TPX_OK;
    if (ck(cudaStreamSynchronize(c->stream))) return TPX_ECUDA;
    if (c->g_mem) cudaFree(c->g_mem);
    c->g_mem = nullptr;
    c->g_bytes = 0;
    if (cudaMalloc(&c->g_mem, bytes) != cudaSuccess) { cudaGetLastError(); return TPX_ENOMEM; }
    c->g_bytes = bytes;
    return TPX_OK;
}

// counts per block of GTILE items -> what the placing kernel expects
int block_prefix(unsigned *bcnt, long long nb, cudaStream_t s) {
    if (nb > kResum) k_scan_bsum<<<1, PT, 0, s>>>(bcnt, nb);
    return ck(cudaGetLastError());
}
inline long long blocks_of(long long n) { return (n + GTILE - 1) / GTILE; }

size_t sort_bytes(long long n) {
    return 2 * sz(n, 8) + 2 * sz(n, 4) + 2 * sz(n, 4) + sz(256 * blocks_of(n), 4) + sz(256, 4) + sz(2, 8) + 4096;
}

// sorts the hits by (shot, corrected ToF); k_seg_count then brings their pixels
// into that order. shot_span >= 0 bounds max shot - min shot (no host round
// trip); < 0 reads it. *pxt_hit: the pixels in hit order.
template <class K>
int sort_keys(tpx_ctx *c, Arena &a, const tpx_hits &h, long long n, int bits, const unsigned long long *mm,
              unsigned *pxt_hit, const K **keys_out, const unsigned **vals_out) {
    cudaStream_t s = c->stream;
    const unsigned tiles = (unsigned)blocks_of(n);
    K *k0 = reinterpret_cast<K *>(a.take<unsigned long long>(n)), *k1 = reinterpret_cast<K *>(a.take<unsigned long long>(n));
    unsigned *v0 = a.take<unsigned>(n), *v1 = a.take<unsigned>(n);
    unsigned *hist = a.take<unsigned>(256ll * tiles), *total = a.take<unsigned>(256);
    constexpr int smem = GTILE * (int)(sizeof(K) + sizeof(unsigned));
    if (ck(cudaFuncSetAttribute(k_digit_place<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return TPX_ECUDA;
    k_make_keys<K><<<tiles, GT, 0, s>>>(h, n, mm, k0, pxt_hit, hist);
    const unsigned *vin = nullptr;   // the first digit's values are the positions themselves
    for (int shift = 0; shift < bits; shift += 8) {
        if (shift > 0) k_digit_hist<K><<<tiles, GT, 0, s>>>(k0, n, shift, hist);
        k_digit_scan<<<256 / 32, PT, 0, s>>>(hist, tiles, total);
        k_digit_place<K><<<tiles, GT, smem, s>>>(k0, vin, n, shift, hist, total, k1, v0);
        vin = v0;
        std::swap(k0, k1);
        std::swap(v0, v1);
    }
    *keys_out = k0;
    *vals_out = vin;
    return ck(cudaGetLastError());
}
int sort_hits(tpx_ctx *c, Arena &a, const tpx_hits &h, long long n, long long shot_span, Sorted *so, unsigned **pxt_hit) {
    cudaStream_t s = c->stream;
    unsigned long long *mm = a.take<unsigned long long>(2);   // min, max shot
    so->pxt = a.take<unsigned>(n);
    *pxt_hit = a.take<unsigned>(n);
    so->hindex = h.index;
    so->shot_min = mm;
    so->k32 = nullptr;
    so->k64 = nullptr;
    if (ck(cudaMemsetAsync(mm, 0xFF, 8, s)) || ck(cudaMemsetAsync(mm + 1, 0, 8, s))) return TPX_ECUDA;
    k_shot_range<<<(unsigned)std::min<long long>((n + 4 * GT - 1) / (4 * GT), (long long)c->num_sms * 4), GT, 0, s>>>(h, n, mm, mm + 1);
    unsigned long long span = (unsigned long long)shot_span;
    if (shot_span < 0) {
        unsigned long long hm[2] = {0, 0};
        if (ck(cudaMemcpyAsync(hm, mm, sizeof hm, cudaMemcpyDeviceToHost, s))) return TPX_ECUDA;
        if (ck(cudaStreamSynchronize(s))) return TPX_ECUDA;
        span = hm[1] - hm[0];
    }
    int bits = 24;
    while (bits < 64 && (span >> (bits - 24)) != 0) ++bits;
    return bits <= 32 ? sort_keys<unsigned>(c, a, h, n, bits, mm, *pxt_hit, &so->k32, &so->hit)
                      : sort_keys<unsigned long long>(c, a, h, n, bits, mm, *pxt_hit, &so->k64, &so->hit);
}

size_t decode_bytes(long long n) {
    const long long tiles = (n + GTILE - 1) / GTILE;
    return sz(tiles, sizeof(GAgg)) * 2 + sz(tiles + 1, 8) * 4 + sz(tiles, 1) + sz(n, 8) + sz(n, 4) + 4096;
}

int decode_impl(tpx_ctx *c, const uint64_t *pk, int64_t n, int64_t base, const tpx_hits &h, int64_t cap,
                int64_t *d_n_hits, int64_t *trig, int64_t trig_cap, int64_t *d_n_trig, bool clear_ctl,
                const GAgg *E0, GAgg *state_out, long long *trig_pos, long long **t_all_out) {
    cudaStream_t s = c->stream;
    const long long tiles = (n + GTILE - 1) / GTILE;
    int rc = reserve(c, decode_bytes(n));
    if (rc) return rc;
    Arena a{static_cast<char *>(c->g_mem), 0, c->g_bytes};
    GAgg *tagg = a.take<GAgg>(tiles), *tpre = a.take<GAgg>(tiles);
    long long *tcnt = a.take<long long>(tiles + 1), *toff = a.take<long long>(tiles + 1);
    long long *tkept = a.take<long long>(tiles + 1), *tkoff = a.take<long long>(tiles + 1);
    unsigned char *twrap = a.take<unsigned char>(tiles);
    long long *t_all = a.take<long long>(n);
    int *shot = a.take<int>(n);
    if (t_all_out) *t_all_out = t_all;
    if (clear_ctl && cudaMemsetAsync(c->ctl, 0, sizeof(Ctl), s) != cudaSuccess) return TPX_ECUDA;
    if (cudaMemsetAsync(d_n_hits, 0, 8, s) != cudaSuccess || cudaMemsetAsync(d_n_trig, 0, 8, s) != cudaSuccess)
        return TPX_ECUDA;
    if (n == 0) {   // the state passes through unchanged
        if (!state_out) return TPX_OK;
        if (E0) return ck(cudaMemcpyAsync(state_out, E0, sizeof(GAgg), cudaMemcpyDeviceToDevice, s));
        return ck(cudaMemsetAsync(state_out, 0, sizeof(GAgg), s));
    }
    const long long tp = c->cfg.wrap_thr_pix_ticks, tt = c->cfg.wrap_thr_tdc_ticks;
    long long *ntr = reinterpret_cast<long long *>(d_n_trig);
    long long *tr = reinterpret_cast<long long *>(trig);
    k_tile_agg<<<(unsigned)tiles, GT, 0, s>>>(pk, n, tp, tt, tagg, tcnt, twrap);
    k_tile_prefix<<<1, PT, 0, s>>>(tagg, tpre, tcnt, toff, tiles, tp, tt, ntr, E0, state_out);
    k_unwrap<<<(unsigned)tiles, GT, 0, s>>>(pk, n, tagg, tpre, twrap, toff, tp, tt, t_all, tr, trig_cap, &c->ctl->status,
                                            trig_pos);
    k_check_trig<<<152, GT, 0, s>>>(tr, ntr, trig_cap, &c->ctl->status);
    k_bin<<<(unsigned)tiles, GT, 0, s>>>(pk, n, t_all, tr, ntr, trig_cap, c->cfg.tof_max_ticks, shot, tkept,
                                         c->ctl->counters);
    k_count_prefix<<<1, PT, 0, s>>>(tkept, tkoff, tiles, reinterpret_cast<long long *>(d_n_hits));
    k_compact<<<(unsigned)tiles, GT, 0, s>>>(pk, n, base, t_all, tr, ntr, trig_cap, shot, c->cfg.d_timewalk_lut, tkoff, h,
                                             cap, &c->ctl->status, E0);
    const unsigned long long np = (unsigned long long)n;
    if (cudaMemcpyAsync(&c->ctl->counters[C_PACKETS], &np, 8, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return TPX_ECUDA;
    return ck(cudaGetLastError());
}

size_t cluster_bytes(long long n) {
    return sort_bytes(n) + sz(n, 4)                                                     // sorted pixels
           + sz(blocks_of(n), 4) + sz(n + 1, 8) + sz(1, 8) + sz(n, 4) + sz(1, 8)         // segments
           + 2 * sz(n, 1) + sz(n, 4)                                                    // long segments
           + sz(n, 1) + sz(n, 4) + sz(n, sizeof(AccH))                                  // records
           + sz(4 * n + 2, 4) + sz(n, 4) + sz(n, 8)                                    // long-segment hash
           + 8192;
}

// The whole clustering stage: sort, segments, labels, local maxima and, when
// `out` is given, the records of the hits whose shot is below shot_limit.
// labels / is_peak (per hit) may be NULL. No host round trip when
// shot_span >= 0.
int cluster_all(tpx_ctx *c, const tpx_hits &h, int64_t n, int64_t *labels, uint8_t *is_peak, long long shot_limit,
                long long shot_span, tpx_record *out, int64_t cap, int64_t *d_n_clusters) {
    cudaStream_t s = c->stream;
    const int cc = c->cfg.mode == TPX_MODE_CC;
    if (out && cudaMemsetAsync(d_n_clusters, 0, 8, s) != cudaSuccess) return TPX_ECUDA;
    if (n <= 0) return TPX_OK;
    int rc = reserve(c, cluster_bytes(n));
    if (rc) return rc;
    Arena a{static_cast<char *>(c->g_mem), 0, c->g_bytes};
    const long long nb = blocks_of(n);
    unsigned *bcnt = a.take<unsigned>(nb), *mid = a.take<unsigned>(n);
    long long *seg_start = a.take<long long>(n + 1), *nseg = a.take<long long>(1);
    SegLists *lists = a.take<SegLists>(1);
    unsigned char *mark = a.take<unsigned char>(n), *notpeak = a.take<unsigned char>(n), *rflag = a.take<unsigned char>(n);
    int *parent = a.take<int>(n);
    unsigned *cid = a.take<unsigned>(n);
    AccH *acc = a.take<AccH>(n);
    unsigned long long lmask = 1;   // the long segments' cell hash: >= 2n buckets
    while (lmask + 1 < 2ull * (unsigned long long)n) lmask = 2 * lmask + 1;
    unsigned *lhead = a.take<unsigned>((long long)lmask + 1), *lnext = a.take<unsigned>(n);
    unsigned long long *lword = a.take<unsigned long long>(n);
    Sorted so;
    unsigned *pxt_hit = nullptr;
    rc = sort_hits(c, a, h, n, shot_span, &so, &pxt_hit);
    if (rc) return rc;
    const int dt = c->cfg.dt_ticks;
    if (ck(cudaMemsetAsync(lists, 0, sizeof(SegLists), s))) return TPX_ECUDA;
    k_seg_count<<<(unsigned)nb, GT, 0, s>>>(so, pxt_hit, n, dt, bcnt);
    rc = block_prefix(bcnt, nb, s);
    if (rc) return rc;
    k_seg_starts<<<(unsigned)nb, GT, 0, s>>>(so, n, dt, bcnt, nb, seg_start, nseg);
    long long *lab = reinterpret_cast<long long *>(labels);
    unsigned char *rf = out ? rflag : nullptr;
    AccH *ac = (out && cc) ? acc : nullptr;
    const long long seg_max = (n + SEGW - 1) / SEGW;   // more blocks than that have no segment
    k_segments<<<(unsigned)std::min<long long>(seg_max, (long long)c->num_sms * 16), SEGW * 32, 0, s>>>(
        so, seg_start, nseg, c->cfg.rx, c->cfg.ry, dt, cc, shot_limit, lab, is_peak, rf, ac, mark, mid, lists);
    // 65 hits at least per block
    k_segments_mid<<<(unsigned)std::min<long long>(n / (WREG + 1) + 1, (long long)c->num_sms * 16), SEGW * 32, 0, s>>>(
        so, seg_start, mid, lists, c->cfg.rx, c->cfg.ry, dt, cc, shot_limit, lab, is_peak, rf, ac);
    k_long_init<<<grid_for(n), GT, 0, s>>>(so, n, lists, mark, parent, notpeak, ac, lhead, lmask);
    k_long_insert<<<grid_for(n), GT, 0, s>>>(so, n, lists, mark, lhead, lnext, lword, lmask);
    k_long_pairs<<<grid_for(n), GT, 0, s>>>(so, n, lists, mark, lhead, lnext, lword, lmask, c->cfg.rx, c->cfg.ry, dt, cc,
                                            parent, notpeak);
    k_long_finish<<<grid_for(n), GT, 0, s>>>(so, n, lists, mark, cc, shot_limit, parent, notpeak, lab, is_peak, rf, ac);
    if (!out) return ck(cudaGetLastError());
    const RootFlag f{nullptr, nullptr, rflag};
    k_root_count<<<(unsigned)nb, GT, 0, s>>>(f, n, bcnt);
    rc = block_prefix(bcnt, nb, s);
    if (rc) return rc;
    const Roots roots{acc, cc ? out : nullptr, cc ? nullptr : cid, nullptr, 0, nullptr, nullptr, nullptr};
    k_root_place<<<(unsigned)nb, GT, 0, s>>>(f, h, n, bcnt, nb, cap, reinterpret_cast<long long *>(d_n_clusters),
                                             &c->ctl->status, &c->ctl->counters[C_CLUSTERS], roots);
    if (!cc) k_paper<<<grid_for(n), GT, 0, s>>>(so, n, c->cfg.rx, c->cfg.ry, dt, rflag, cid, h, out, cap);
    return ck(cudaGetLastError());
}

int cluster_impl(tpx_ctx *c, const tpx_hits &h, int64_t n, int64_t *labels, uint8_t *is_peak) {
    return cluster_all(c, h, n, labels, is_peak, LLONG_MAX, -1, nullptr, 0, nullptr);
}

int centroid_impl(tpx_ctx *c, const tpx_hits &h, const int64_t *labels, const uint8_t *is_peak, int64_t n,
                  tpx_record *out, int64_t cap, int64_t *d_n_clusters) {
    cudaStream_t s = c->stream;
    if (ck(cudaMemsetAsync(d_n_clusters, 0, 8, s))) return TPX_ECUDA;
    if (n <= 0) return TPX_OK;
    const int cc = c->cfg.mode == TPX_MODE_CC;
    if (!cc && !is_peak) return TPX_EINVAL;
    const long long nb = blocks_of(n);
    const long long recs = std::min<long long>(n, cap), rank_cap = 2 * n + 65536;
    const size_t need = sz(nb, 4) + (cc ? sz(rank_cap, 4) + sz(recs, sizeof(Acc)) + sz(recs, 4) + sz(recs, 8)
                                        : sz(n, 4) + sz(n, 4) + sort_bytes(n)) + 8192;
    int rc = reserve(c, need);
    if (rc) return rc;
    Arena a{static_cast<char *>(c->g_mem), 0, c->g_bytes};
    unsigned *bcnt = a.take<unsigned>(nb);
    const long long *lab = reinterpret_cast<const long long *>(labels);
    long long *nrec = reinterpret_cast<long long *>(d_n_clusters);
    const RootFlag f{cc ? lab : nullptr, reinterpret_cast<const long long *>(h.index), cc ? nullptr : is_peak};
    k_root_count<<<(unsigned)nb, GT, 0, s>>>(f, n, bcnt);
    rc = block_prefix(bcnt, nb, s);
    if (rc) return rc;
    if (cc) {
        unsigned *rank = a.take<unsigned>(rank_cap), *rootpos = a.take<unsigned>(recs);
        Acc *acc = a.take<Acc>(recs);
        long long *root_t = a.take<long long>(recs);
        if (ck(cudaMemsetAsync(rank, 0xFF, 4 * (size_t)rank_cap, s))) return TPX_ECUDA;
        const Roots roots{nullptr, nullptr, nullptr, rank, rank_cap, acc, rootpos, root_t};
        k_root_place<<<(unsigned)nb, GT, 0, s>>>(f, h, n, bcnt, nb, cap, nrec, &c->ctl->status,
                                                 &c->ctl->counters[C_CLUSTERS], roots);
        k_accum<<<(unsigned)nb, GT, 0, s>>>(h, lab, is_peak, n, nrec, cap, rank, rank_cap, rootpos, root_t, acc);
        k_final<<<grid_for(recs / 8 + 1), GT, 0, s>>>(h, nrec, cap, rootpos, acc, out);
    } else {
        unsigned *cid = a.take<unsigned>(n);
        const Roots roots{nullptr, nullptr, cid, nullptr, 0, nullptr, nullptr, nullptr};
        k_root_place<<<(unsigned)nb, GT, 0, s>>>(f, h, n, bcnt, nb, cap, nrec, &c->ctl->status,
                                                 &c->ctl->counters[C_CLUSTERS], roots);
        Sorted so;
        unsigned *pxt_hit = nullptr;
        rc = sort_hits(c, a, h, n, -1, &so, &pxt_hit);
        if (rc) return rc;
        k_seg_count<<<(unsigned)nb, GT, 0, s>>>(so, pxt_hit, n, c->cfg.dt_ticks, bcnt);   // brings the pixels into order
        k_paper<<<grid_for(n), GT, 0, s>>>(so, n, c->cfg.rx, c->cfg.ry, c->cfg.dt_ticks, is_peak, cid, h, out, cap);
    }
    return ck(cudaGetLastError());
}

__global__ void k_packet_outputs(tpx_hits h, const long long *hl, const unsigned char *hp, long long nh, long long base,
                                 long long *labels, unsigned char *is_peak) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nh; i += (long long)gridDim.x * blockDim.x) {
        const long long q = h.index[i] - base;
        if (labels) labels[q] = hl[i];
        if (is_peak) is_peak[q] = hp[i];
    }
}
__global__ void k_packet_labels32(tpx_hits h, const long long *hl, long long nh, long long base, long long lbase,
                                  int *labels) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nh; i += (long long)gridDim.x * blockDim.x)
        labels[h.index[i] - base] = (int)(hl[i] - lbase);
}
__global__ void k_fill_i32(int *p, long long n, int v) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) p[i] = v;
}
__global__ void k_records64(const tpx_record *src, const long long *n, long long cap, tpx_record64 *dst) {
    const long long m = min(*n, cap);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < m; i += (long long)gridDim.x * blockDim.x)
        dst[i] = *reinterpret_cast<const tpx_record64 *>(src + i);
}
__global__ void k_fill_ll(long long *p, long long n, long long v) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) p[i] = v;
}
__global__ void k_count_peaks(const unsigned char *hp, long long n, unsigned long long *cnt) {
    unsigned long long m = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) m += hp[i];
    for (int o = 16; o > 0; o >>= 1) m += __shfl_down_sync(0xffffffffu, m, o);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(cnt, m);
}

int redo_last(tpx_ctx *c) {
    if (!c->last.valid) return TPX_EINVAL;
    const auto L = c->last;
    const long long n = L.n;
    if (n >= (1LL << 31)) return TPX_EUNSUPPORTED;
    cudaStream_t s = c->stream;
    // hits and per-hit outputs live in a separate allocation from the arena
    // used by the stages (each stage reuses the arena from its start)
    const size_t hb = sz(n, 8) * 4 + sz(n, 4) + 3 * sz(n, 2) + sz(n, 1) * 3 + 4096;
    void *hm = nullptr;
    if (cudaMalloc(&hm, hb) != cudaSuccess) { cudaGetLastError(); return TPX_ENOMEM; }
    Arena a{static_cast<char *>(hm), 0, hb};
    tpx_hits h;
    h.index = reinterpret_cast<int64_t *>(a.take<long long>(n));
    h.shot = reinterpret_cast<int64_t *>(a.take<long long>(n));
    h.t = reinterpret_cast<int64_t *>(a.take<long long>(n));
    h.tof = a.take<int32_t>(n);
    h.x = a.take<uint8_t>(n);
    h.y = a.take<uint8_t>(n);
    h.tot = a.take<uint16_t>(n);
    long long *hl = a.take<long long>(n);
    unsigned char *hp = a.take<unsigned char>(n);
    long long *nh_d = a.take<long long>(1);
    int rc = decode_impl(c, L.pk, n, L.base, h, n, reinterpret_cast<int64_t *>(nh_d), L.trig, L.trig_cap, L.n_trig, true,
                         L.E0, L.state_out, nullptr, nullptr);
    long long nh = 0;
    if (!rc) rc = ck(cudaMemcpyAsync(&nh, nh_d, 8, cudaMemcpyDeviceToHost, s));
    if (!rc) rc = ck(cudaStreamSynchronize(s));
    unsigned status = 0;
    if (!rc) rc = ck(cudaMemcpy(&status, &c->ctl->status, 4, cudaMemcpyDeviceToHost));
    if (!rc && !(status & (ST_TRIG_ORDER | ST_TRIG_CAP))) {
        // TPX_FLAG_RECORDS64: the full records go to a scratch array first,
        // then their first 64 bytes to the caller's buffer
        const bool r64 = (c->cfg.flags & TPX_FLAG_RECORDS64) != 0 && L.cl_cap > 0;
        const int64_t cap64 = r64 ? std::min<int64_t>(L.cl_cap, std::max<long long>(nh, 1)) : 0;
        tpx_record *out = L.cl;
        void *tmp = nullptr;
        if (r64) {
            if (cudaMalloc(&tmp, sizeof(tpx_record) * (size_t)cap64) != cudaSuccess) { cudaGetLastError(); rc = TPX_ENOMEM; }
            out = static_cast<tpx_record *>(tmp);
        }
        if (!rc) rc = cluster_all(c, h, nh, reinterpret_cast<int64_t *>(hl), hp, LLONG_MAX, -1, out, r64 ? cap64 : L.cl_cap,
                                  L.n_cl);
        if (!rc && r64) {
            k_records64<<<grid_for(cap64), GT, 0, s>>>(static_cast<const tpx_record *>(tmp), reinterpret_cast<const long long *>(L.n_cl),
                                                     cap64, reinterpret_cast<tpx_record64 *>(L.cl));
            rc = ck(cudaStreamSynchronize(s));
        }
        if (tmp) cudaFree(tmp);
        if (!rc && (L.labels || L.is_peak)) {
            long long *l64 = L.lab32 ? nullptr : reinterpret_cast<long long *>(L.labels);
            int *l32 = L.lab32 ? reinterpret_cast<int *>(L.labels) : nullptr;
            if (l64) k_fill_ll<<<grid_for(n), GT, 0, s>>>(l64, n, -1);
            if (l32) k_fill_i32<<<grid_for(n), GT, 0, s>>>(l32, n, -1);
            if (L.is_peak && cudaMemsetAsync(L.is_peak, 0, (size_t)n, s) != cudaSuccess) rc = TPX_ECUDA;
            k_packet_outputs<<<grid_for(nh), GT, 0, s>>>(h, hl, hp, nh, L.base, l64, L.is_peak);
            if (l32) k_packet_labels32<<<grid_for(nh), GT, 0, s>>>(h, hl, nh, L.base, L.lab32_base, l32);
        }
        if (!rc && nh > 0) {
            unsigned long long z = 0;
            rc = ck(cudaMemcpyAsync(&c->ctl->counters[C_PEAKS], &z, 8, cudaMemcpyHostToDevice, s));
            k_count_peaks<<<grid_for(nh), GT, 0, s>>>(hp, nh, &c->ctl->counters[C_PEAKS]);
        }
    }
    if (!rc) {
        // the counters now describe the redone call
        unsigned long long np = (unsigned long long)n;
        rc = ck(cudaMemcpyAsync(&c->ctl->counters[C_PACKETS], &np, 8, cudaMemcpyHostToDevice, s));
    }
    if (!rc) rc = ck(cudaStreamSynchronize(s));
    cudaFree(hm);
    return rc;
}

// ---- redo of a batch's failed runs ----
__global__ void k_add_ll(long long *v, long long n, long long d) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        v[i] += d;
}
// first record of each run of a group: records are in label order and the
// runs' labels are the runs' packet ranges
__global__ void k_rec_bounds(const tpx_record *rec, long long ncl, const long long *run_start, long long nr,
                             long long *bound) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k <= nr; k += (long long)gridDim.x * blockDim.x) {
        if (k == nr) { bound[k] = ncl; continue; }
        long long lo = 0, hi = ncl;
        while (lo < hi) {
            const long long mid = lo + ((hi - lo) >> 1);
            if (rec[mid].label < run_start[k]) lo = mid + 1; else hi = mid;
        }
        bound[k] = lo;
    }
}
// records of group run k count their shots from the run's first trigger
__global__ void k_rec_shots(tpx_record *rec, long long ncl, const long long *bound, const long long *shot_base,
                            long long nr) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ncl; i += (long long)gridDim.x * blockDim.x) {
        long long lo = 0, hi = nr;   // the run k with bound[k] <= i < bound[k + 1]
        while (hi - lo > 1) {
            const long long mid = (lo + hi) >> 1;
            if (bound[mid] <= i) lo = mid; else hi = mid;
        }
        rec[i].shot -= shot_base[lo];
    }
}
// segmented copy of 8-byte words: segment i moves len[i] words src[i] -> dst[i]
__global__ void k_seg_copy(const unsigned long long *const *src, unsigned long long *const *dst, const long long *len,
                           long long nseg) {
    for (long long i = blockIdx.x; i < nseg; i += gridDim.x) {
        const unsigned long long *a = src[i];
        unsigned long long *b = dst[i];
        for (long long w = threadIdx.x; w < len[i]; w += blockDim.x) b[w] = a[w];
    }
}

namespace {
// a device buffer that keeps its contents when it grows
struct Grow {
    char *p = nullptr;
    size_t used = 0, cap = 0;
    int ensure(size_t want, cudaStream_t s) {
        if (want <= cap) return TPX_OK;
        size_t nc = cap ? cap : (size_t)1 << 24;
        while (nc < want) nc *= 2;
        char *q = nullptr;
        if (cudaMalloc(&q, nc) != cudaSuccess) { cudaGetLastError(); return TPX_ENOMEM; }
        if (used && ck(cudaMemcpyAsync(q, p, used, cudaMemcpyDeviceToDevice, s))) { cudaFree(q); return TPX_ECUDA; }
        if (ck(cudaStreamSynchronize(s))) { cudaFree(q); return TPX_ECUDA; }
        if (p) cudaFree(p);
        p = q;
        cap = nc;
        return TPX_OK;
    }
    ~Grow() { if (p) cudaFree(p); }
};
}  // namespace

int redo_batch(tpx_ctx *c, int64_t *n_redone) {
    auto &B = c->batch;
    cudaStream_t s = c->stream;
    const int64_t R = B.n_runs;
    const int64_t *off = B.h_off;   // the run offsets of the call (host)
    *n_redone = 0;
    std::vector<unsigned> failed((size_t)R);
    std::vector<int64_t> roff((size_t)R + 1), toff((size_t)R + 1);
    Ctl snap;
    if (ck(cudaMemcpyAsync(failed.data(), B.bt.run_failed, 4 * (size_t)R, cudaMemcpyDeviceToHost, s)) ||
        ck(cudaMemcpyAsync(roff.data(), B.bt.run_rec_off, 8 * (size_t)(R + 1), cudaMemcpyDeviceToHost, s)) ||
        ck(cudaMemcpyAsync(toff.data(), B.bt.run_trig_off, 8 * (size_t)(R + 1), cudaMemcpyDeviceToHost, s)) ||
        ck(cudaMemcpyAsync(&snap, c->ctl, sizeof snap, cudaMemcpyDeviceToHost, s)))
        return TPX_ECUDA;
    if (ck(cudaStreamSynchronize(s))) return TPX_ECUDA;
    // the tiles' pass wrote records and triggers only below the capacities
    for (int64_t r = 0; r <= R; ++r) {
        roff[(size_t)r] = std::min<int64_t>(roff[(size_t)r], B.cl_cap);
        toff[(size_t)r] = std::min<int64_t>(toff[(size_t)r], B.trig_cap);
    }
    std::vector<int64_t> F;
    int64_t max_len = 0;
    for (int64_t r = 0; r < R; ++r)
        if (failed[(size_t)r]) {
            F.push_back(r);
            max_len = std::max<int64_t>(max_len, off[r + 1] - off[r]);
        }
    *n_redone = (int64_t)F.size();
    if (F.empty()) return TPX_OK;
    // failed runs are redone in groups of consecutive failed runs holding at
    // most G packets (or one larger run): each run decodes on its own (a
    // stream of its own), its shots offset to keep the group's shots apart,
    // and one clustering pass serves the whole group
    const int64_t G = std::max<int64_t>(max_len, 1LL << 26);
    if (G >= (1LL << 31)) return TPX_EUNSUPPORTED;
    const bool per_packet = B.labels || B.is_peak;
    const size_t hb = sz(G, 8) * 3 + sz(G, 4) + sz(G, 2) + 2 * sz(G, 1) + (per_packet ? sz(G, 8) + sz(G, 1) : 0) +
                      sz(G, 8) + sz(G, sizeof(tpx_record)) + 3 * sz((int64_t)F.size() + 1, 8) + sz(4, 8) + 4096;
    void *hm = nullptr;
    if (cudaMalloc(&hm, hb) != cudaSuccess) { cudaGetLastError(); return TPX_ENOMEM; }
    Arena a{static_cast<char *>(hm), 0, hb};
    tpx_hits h;
    h.index = reinterpret_cast<int64_t *>(a.take<long long>(G));
    h.shot = reinterpret_cast<int64_t *>(a.take<long long>(G));
    h.t = reinterpret_cast<int64_t *>(a.take<long long>(G));
    h.tof = a.take<int32_t>(G);
    h.tot = a.take<uint16_t>(G);
    h.x = a.take<uint8_t>(G);
    h.y = a.take<uint8_t>(G);
    long long *hl = per_packet ? a.take<long long>(G) : nullptr;
    unsigned char *hp = per_packet ? a.take<unsigned char>(G) : nullptr;
    long long *tr = a.take<long long>(G);
    tpx_record *grec = a.take<tpx_record>(G);
    long long *d_start = a.take<long long>((int64_t)F.size() + 1), *d_base = a.take<long long>((int64_t)F.size() + 1);
    long long *d_bound = a.take<long long>((int64_t)F.size() + 1);
    long long *cnt = a.take<long long>(4);
    Grow acc_rec, acc_trig;   // the redone runs' records and triggers, run after run
    std::vector<int64_t> nrec((size_t)R), ntrg((size_t)R), rstart((size_t)R), tstart((size_t)R);
    int rc = TPX_OK;
    for (size_t i = 0; i < F.size() && !rc;) {
        size_t j = i;
        int64_t pk_sum = 0;
        while (j < F.size() && (j == i || pk_sum + (off[F[j] + 1] - off[F[j]]) <= G)) {
            pk_sum += off[F[j] + 1] - off[F[j]];
            ++j;
        }
        const int64_t nr = (int64_t)(j - i);
        std::vector<long long> start((size_t)nr), base((size_t)nr);
        int64_t hoff = 0, tcount = 0;
        for (int64_t k = 0; k < nr && !rc; ++k) {
            const int64_t r = F[i + (size_t)k], len = off[r + 1] - off[r];
            tpx_hits hk = h;
            hk.index += hoff; hk.shot += hoff; hk.t += hoff; hk.tof += hoff; hk.tot += hoff; hk.x += hoff; hk.y += hoff;
            rc = decode_impl(c, B.pk + off[r], len, off[r], hk, len, reinterpret_cast<int64_t *>(cnt),
                             reinterpret_cast<int64_t *>(tr + tcount), len, reinterpret_cast<int64_t *>(cnt + 1), false,
                             nullptr, nullptr, nullptr, nullptr);
            long long hc[2] = {0, 0};
            if (!rc) rc = ck(cudaMemcpyAsync(hc, cnt, 16, cudaMemcpyDeviceToHost, s));
            if (!rc) rc = ck(cudaStreamSynchronize(s));
            if (rc) break;
            if (hc[0] > 0 && tcount > 0) k_add_ll<<<grid_for(hc[0]), GT, 0, s>>>(reinterpret_cast<long long *>(hk.shot), hc[0], tcount);
            start[(size_t)k] = off[r];
            base[(size_t)k] = tcount;
            ntrg[(size_t)r] = hc[1];
            hoff += hc[0];
            tcount += hc[1];
        }
        if (rc) break;
        // one clustering pass for the group; records in label order = run order
        rc = cluster_all(c, h, hoff, reinterpret_cast<int64_t *>(hl), hp, LLONG_MAX, tcount, grec, hoff,
                         reinterpret_cast<int64_t *>(cnt + 2));
        if (!rc && per_packet && hoff > 0) {
            for (int64_t k = 0; k < nr; ++k) {
                const int64_t r = F[i + (size_t)k], len = off[r + 1] - off[r];
                if (B.labels) k_fill_ll<<<grid_for(len), GT, 0, s>>>(reinterpret_cast<long long *>(B.labels) + off[r], len, -1);
                if (B.is_peak && ck(cudaMemsetAsync(B.is_peak + off[r], 0, (size_t)len, s))) rc = TPX_ECUDA;
            }
            k_packet_outputs<<<grid_for(hoff), GT, 0, s>>>(h, hl, hp, hoff, 0, reinterpret_cast<long long *>(B.labels),
                                                           B.is_peak);
        }
        long long ncl = 0;
        if (!rc) rc = ck(cudaMemcpyAsync(&ncl, cnt + 2, 8, cudaMemcpyDeviceToHost, s));
        if (!rc) rc = ck(cudaMemcpyAsync(d_start, start.data(), 8 * (size_t)nr, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(d_base, base.data(), 8 * (size_t)nr, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaStreamSynchronize(s));
        if (rc) break;
        if (hoff == 0) ncl = 0;
        std::vector<long long> bound((size_t)nr + 1, 0);
        if (ncl > 0) {
            k_rec_bounds<<<grid_for(nr + 1), GT, 0, s>>>(grec, ncl, d_start, nr, d_bound);
            k_rec_shots<<<grid_for(ncl), GT, 0, s>>>(grec, ncl, d_bound, d_base, nr);
            rc = ck(cudaMemcpyAsync(bound.data(), d_bound, 8 * (size_t)(nr + 1), cudaMemcpyDeviceToHost, s));
        }
        // append the group's records and triggers
        if (!rc) rc = acc_rec.ensure(acc_rec.used + sizeof(tpx_record) * (size_t)ncl, s);
        if (!rc) rc = acc_trig.ensure(acc_trig.used + 8 * (size_t)tcount, s);
        if (!rc && ncl > 0)
            rc = ck(cudaMemcpyAsync(acc_rec.p + acc_rec.used, grec, sizeof(tpx_record) * (size_t)ncl,
                                    cudaMemcpyDeviceToDevice, s));
        if (!rc && tcount > 0)
            rc = ck(cudaMemcpyAsync(acc_trig.p + acc_trig.used, tr, 8 * (size_t)tcount, cudaMemcpyDeviceToDevice, s));
        if (!rc) rc = ck(cudaStreamSynchronize(s));
        if (rc) break;
        for (int64_t k = 0; k < nr; ++k) {
            const int64_t r = F[i + (size_t)k];
            nrec[(size_t)r] = bound[(size_t)k + 1] - bound[(size_t)k];
            rstart[(size_t)r] = (int64_t)(acc_rec.used / sizeof(tpx_record)) + bound[(size_t)k];
            tstart[(size_t)r] = (int64_t)(acc_trig.used / 8) + base[(size_t)k];
        }
        acc_rec.used += sizeof(tpx_record) * (size_t)ncl;
        acc_trig.used += 8 * (size_t)tcount;
        i = j;
    }
    // the runs' final offsets; every run from the first redone one on moves
    // (the tiles' outputs of the others are kept aside first)
    const int64_t first = F.front();
    std::vector<long long> NO((size_t)R + 1), NTo((size_t)R + 1);
    NO[0] = 0;
    NTo[0] = 0;
    for (int64_t r = 0; r < R; ++r) {
        NO[(size_t)r + 1] = NO[(size_t)r] + (failed[(size_t)r] ? nrec[(size_t)r] : roff[(size_t)r + 1] - roff[(size_t)r]);
        NTo[(size_t)r + 1] = NTo[(size_t)r] + (failed[(size_t)r] ? ntrg[(size_t)r] : toff[(size_t)r + 1] - toff[(size_t)r]);
    }
    const int64_t old_rec = roff[(size_t)R] - roff[(size_t)first], old_trig = toff[(size_t)R] - toff[(size_t)first];
    Grow keep;
    if (!rc) rc = keep.ensure(sizeof(tpx_record) * (size_t)old_rec + 8 * (size_t)old_trig + 512, s);
    tpx_record *old_rec_copy = reinterpret_cast<tpx_record *>(keep.p);
    long long *old_trig_copy = reinterpret_cast<long long *>(keep.p + ((sizeof(tpx_record) * (size_t)old_rec + 255) & ~size_t(255)));
    if (!rc && old_rec > 0)
        rc = ck(cudaMemcpyAsync(old_rec_copy, B.cl + roff[(size_t)first], sizeof(tpx_record) * (size_t)old_rec,
                                cudaMemcpyDeviceToDevice, s));
    if (!rc && old_trig > 0)
        rc = ck(cudaMemcpyAsync(old_trig_copy, B.trig + toff[(size_t)first], 8 * (size_t)old_trig, cudaMemcpyDeviceToDevice, s));
    // one segmented copy for all moved runs (records, then triggers)
    std::vector<const unsigned long long *> src;
    std::vector<unsigned long long *> dst;
    std::vector<long long> len;
    constexpr int WPR = (int)(sizeof(tpx_record) / 8);
    for (int64_t r = first; r < R && !rc; ++r) {
        const int64_t nr = NO[(size_t)r + 1] - NO[(size_t)r], nt = NTo[(size_t)r + 1] - NTo[(size_t)r];
        const int64_t kr = std::max<int64_t>(0, std::min<int64_t>(nr, B.cl_cap - NO[(size_t)r]));
        const int64_t kt = std::max<int64_t>(0, std::min<int64_t>(nt, B.trig_cap - NTo[(size_t)r]));
        const tpx_record *sr = failed[(size_t)r] ? reinterpret_cast<const tpx_record *>(acc_rec.p) + rstart[(size_t)r]
                                                 : old_rec_copy + (roff[(size_t)r] - roff[(size_t)first]);
        const long long *st = failed[(size_t)r] ? reinterpret_cast<const long long *>(acc_trig.p) + tstart[(size_t)r]
                                                : old_trig_copy + (toff[(size_t)r] - toff[(size_t)first]);
        if (kr > 0) {
            src.push_back(reinterpret_cast<const unsigned long long *>(sr));
            dst.push_back(reinterpret_cast<unsigned long long *>(B.cl + NO[(size_t)r]));
            len.push_back(kr * WPR);
        }
        if (kt > 0) {
            src.push_back(reinterpret_cast<const unsigned long long *>(st));
            dst.push_back(reinterpret_cast<unsigned long long *>(B.trig + NTo[(size_t)r]));
            len.push_back(kt);
        }
    }
    if (!rc && !len.empty()) {
        {   // pieces of at most 2^16 words, so that large runs spread over blocks
            std::vector<const unsigned long long *> s2;
            std::vector<unsigned long long *> d2;
            std::vector<long long> l2;
            for (size_t k = 0; k < len.size(); ++k)
                for (long long o = 0; o < len[k]; o += 1 << 16) {
                    s2.push_back(src[k] + o);
                    d2.push_back(dst[k] + o);
                    l2.push_back(std::min<long long>(1 << 16, len[k] - o));
                }
            src.swap(s2);
            dst.swap(d2);
            len.swap(l2);
        }
        const size_t ns = len.size();
        Grow desc;
        rc = desc.ensure(3 * 8 * ns + 512, s);
        void **d_src = reinterpret_cast<void **>(desc.p);
        void **d_dst = d_src + ns;
        long long *d_len = reinterpret_cast<long long *>(d_dst + ns);
        if (!rc) rc = ck(cudaMemcpyAsync(d_src, src.data(), 8 * ns, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(d_dst, dst.data(), 8 * ns, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(d_len, len.data(), 8 * ns, cudaMemcpyHostToDevice, s));
        if (!rc)
            k_seg_copy<<<(unsigned)std::min<size_t>(ns, 152 * 8), 256, 0, s>>>(
                reinterpret_cast<const unsigned long long *const *>(d_src), reinterpret_cast<unsigned long long *const *>(d_dst),
                d_len, (long long)ns);
        if (!rc) rc = ck(cudaStreamSynchronize(s));   // the descriptors are freed on return
    }
    if (!rc) {
        // offsets, totals; the counters keep describing the tiles' pass
        snap.counters[C_CLUSTERS] = (unsigned long long)NO[(size_t)R];
        if (NO[(size_t)R] > B.cl_cap) snap.status |= ST_CLUSTER_CAP;
        if (NTo[(size_t)R] > B.trig_cap) snap.status |= ST_TRIG_CAP;
        Ctl cur;
        rc = ck(cudaMemcpyAsync(&cur, c->ctl, sizeof cur, cudaMemcpyDeviceToHost, s));
        if (!rc) rc = ck(cudaStreamSynchronize(s));
        snap.status |= cur.status & ST_TRIG_ORDER;   // a redone run may have decreasing triggers
        snap.status &= ~ST_RUN_REDO;                 // done: a later sync has nothing to redo
        if (!rc) rc = ck(cudaMemcpyAsync(B.bt.run_rec_off, NO.data(), 8 * (size_t)(R + 1), cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(B.bt.run_trig_off, NTo.data(), 8 * (size_t)(R + 1), cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(B.n_cl, &NO[(size_t)R], 8, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(B.n_trig, &NTo[(size_t)R], 8, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaMemcpyAsync(c->ctl, &snap, sizeof snap, cudaMemcpyHostToDevice, s));
        if (!rc) rc = ck(cudaStreamSynchronize(s));
    }
    cudaStreamSynchronize(s);
    cudaFree(hm);
    return rc;
}

}  // namespace tpxg

// ------------------------------------------------------------ C ABI
extern "C" int tpx_decode(tpx_ctx *c, const uint64_t *pk, int64_t n, int64_t base, const tpx_hits *hits,
                          int64_t cap, int64_t *d_n_hits, int64_t *trig, int64_t trig_cap, int64_t *d_n_trig) {
    if (!c || !hits || n < 0 || cap < 0 || trig_cap < 0 || !d_n_hits || !d_n_trig) return TPX_EINVAL;
    if (n > 0 && !pk) return TPX_EINVAL;
    if (n >= (1LL << 31)) return TPX_EINVAL;
    if (cap > 0 && (!hits->index || !hits->shot || !hits->t || !hits->tof || !hits->x || !hits->y || !hits->tot))
        return TPX_EINVAL;
    if (trig_cap > 0 && !trig) return TPX_EINVAL;
    c->last.valid = false;
    const tpxk::GAgg *E0 = nullptr;
    tpxk::GAgg *out = nullptr;
    take_state(c, &E0, &out);
    return tpxg::decode_impl(c, pk, n, base, *hits, cap, d_n_hits, trig, trig_cap, d_n_trig, true, E0, out, nullptr,
                             nullptr);
}

extern "C" int tpx_cluster(tpx_ctx *c, const tpx_hits *hits, int64_t n, int64_t *d_labels, uint8_t *d_is_peak) {
    if (!c || !hits || n < 0 || n >= (1LL << 31) || (n > 0 && !d_labels)) return TPX_EINVAL;
    c->last.valid = false;
    return tpxg::cluster_impl(c, *hits, n, d_labels, d_is_peak);
}

extern "C" int tpx_centroid(tpx_ctx *c, const tpx_hits *hits, const int64_t *d_labels, const uint8_t *d_is_peak,
                            int64_t n, tpx_record *d_clusters, int64_t cap, int64_t *d_n_clusters) {
    if (!c || !hits || n < 0 || n >= (1LL << 31) || cap < 0 || !d_n_clusters) return TPX_EINVAL;
    if ((n > 0 && !d_labels) || (cap > 0 && !d_clusters)) return TPX_EINVAL;
    c->last.valid = false;
    return tpxg::centroid_impl(c, *hits, d_labels, d_is_peak, n, d_clusters, cap, d_n_clusters);
}

namespace tpxg {
// one count per hit inside the ToF window (Sec. IV.C calibration histogram)
__global__ void k_tot_tof_hist(const int32_t *tof, const uint16_t *tot, long long n, int lo, int bin, int nb,
                               unsigned *hist) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long d = (long long)tof[i] - lo;
        if (d < 0) continue;
        const long long b = d / bin;
        if (b >= nb) continue;
        atomicAdd(&hist[(long long)tot[i] * nb + b], 1u);
    }
}
}  // namespace tpxg

extern "C" int tpx_tot_tof_histogram(tpx_ctx *c, const tpx_hits *hits, int64_t n, int32_t lo, int32_t bin, int32_t nb,
                                     uint32_t *d_hist) {
    if (!c || !hits || n < 0 || bin < 1 || nb < 1 || !d_hist) return TPX_EINVAL;
    if (n > 0 && (!hits->tof || !hits->tot)) return TPX_EINVAL;
    if (n == 0) return TPX_OK;
    tpxg::k_tot_tof_hist<<<tpxg::grid_for(n), tpxg::GT, 0, c->stream>>>(hits->tof, hits->tot, n, lo, bin, nb, d_hist);
    return tpxg::ck(cudaGetLastError());
}

extern "C" int tpx_summarize(tpx_ctx *c, const uint64_t *pk, int64_t n, tpx_chain_summary *out) {
    if (!c || !out || n < 0 || (n > 0 && !pk)) return TPX_EINVAL;
    using namespace tpxg;
    cudaStream_t s = c->stream;
    const long long tiles = (n + GTILE - 1) / GTILE;
    const size_t need = sz(tiles, sizeof(tpxk::GAgg)) * 2 + sz(tiles + 1, 8) * 2 + sz(1, sizeof(tpxk::GAgg)) + sz(tiles, 1) + 4096;
    int rc = reserve(c, need);
    if (rc) return rc;
    Arena a{static_cast<char *>(c->g_mem), 0, c->g_bytes};
    tpxk::GAgg *tagg = a.take<tpxk::GAgg>(tiles), *tpre = a.take<tpxk::GAgg>(tiles);
    long long *tcnt = a.take<long long>(tiles + 1), *toff = a.take<long long>(tiles + 1);
    tpxk::GAgg *res = a.take<tpxk::GAgg>(1);
    unsigned char *twrap = a.take<unsigned char>(tiles);
    long long *ntr = toff + tiles;
    tpxk::GAgg h;
    std::memset(&h, 0, sizeof h);
    if (n > 0) {
        const long long tp = c->cfg.wrap_thr_pix_ticks, tt = c->cfg.wrap_thr_tdc_ticks;
        k_tile_agg<<<(unsigned)tiles, GT, 0, s>>>(pk, n, tp, tt, tagg, tcnt, twrap);
        k_tile_prefix<<<1, PT, 0, s>>>(tagg, tpre, tcnt, toff, tiles, tp, tt, ntr, nullptr, res);
        if (ck(cudaMemcpyAsync(&h, res, sizeof h, cudaMemcpyDeviceToHost, s))) return TPX_ECUDA;
    }
    if (ck(cudaStreamSynchronize(s))) return TPX_ECUDA;
    out->pixels = h.pix.n;
    out->pix_first_raw = h.pix.first;
    out->pix_last_raw = h.pix.last;
    out->pix_wraps = h.pix.sum;
    out->triggers = h.tdc.n;
    out->tdc_first_raw = h.tdc.first;
    out->tdc_last_raw = h.tdc.last;
    out->tdc_wraps = h.tdc.sum;
    return TPX_OK;
}
