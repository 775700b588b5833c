// tpx_prepass.cu -- the unwrap state before every tile of the fused kernel.
//
// ToA unwrapping (Sec. IV.A) is a chain along each of the two streams (pixels,
// TDCs): a step down by more than the threshold adds a wrap, a step up by more
// removes one. The fused kernel needs, for each tile of packets it claims, the
// chain state where the tile starts: the wraps counted so far, the raw value
// of the last pixel and TDC packet before it, and the number of triggers
// before it (the shot index base). This pass computes those states ahead of
// the fused kernel, so that a tile never waits for its predecessors:
//   1. k_tile_aggs: one warp per tile reads the tile once (coalesced 16-byte
//      loads) and forms the tile's chain aggregate (count, first and last raw
//      value, wraps inside) of each stream. Wraps are rare, so the steps are
//      found lane by lane with ballots instead of a scan per load;
//   2. k_block_scan: an exclusive scan of the tile aggregates inside blocks of
//      1024 tiles, and each block's total;
//   3. k_top_scan: one block scans the block totals, starting from the state
//      before the call;
//   4. k_apply: the state before each tile (its pixel chain carried on to the
//      tile's first TDC packet, where the tile's range starts), and after the
//      last one.
// Up to 1024 tiles one launch does all of it (k_prepass_small).
// Beside the aggregates, k_tile_aggs leaves what the fused kernel plans its
// ranges from (TileInfo): each tile's first TDC packet and whether a pixel wrap
// lies in it, so that the fused kernel neither searches for the end of a range
// nor follows the pixel chain inside it, save near a wrap.
// In a batch of independent runs every run is a stream of its own: the scan is
// segmented, restarting at each run's first tile.
#include <cuda_runtime.h>

#include <cstdint>

#include "tpx_common.cuh"
#include "tpx_fused.cuh"
#include "tpx_unwrap.cuh"

namespace tpxk {
namespace {

constexpr int SB = 1024;       // tiles per block of the scan
constexpr int AW = 8;          // warps per block of k_tile_aggs

// the packets of a tile: [base, base + cnt), and whether a run starts there
struct TileSpan { long long base; int cnt; bool run_first; };
__device__ __forceinline__ TileSpan tile_span(const Params &p, long long tile, int T) {
    TileSpan s;
    long long rend = p.n;
    if (p.bt.tile_run) {
        const int run = p.bt.tile_run[tile];
        const long long t0 = p.bt.run_tile0[run];
        s.base = p.bt.run_off[run] + (tile - t0) * T;
        rend = p.bt.run_off[run + 1];
        s.run_first = tile == t0;
    } else {
        s.base = tile * T;
        s.run_first = tile == 0;
    }
    s.cnt = (int)max(0LL, min((long long)T, rend - s.base));
    return s;
}

__global__ void __launch_bounds__(AW * 32, 3) k_tile_aggs(const Params p, int T) {
    const int lane = threadIdx.x & 31;
    const long long warp = (long long)blockIdx.x * AW + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * AW;
    unsigned long long c_pix = 0, c_tdc = 0, c_bad = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {   // the fused kernel's last tile writes them
        *p.n_clusters = 0;
        *p.n_trig = 0;
    }
    for (long long tile = warp; tile < p.n_tiles; tile += nw) {
        const TileSpan sp = tile_span(p, tile, T);
        WarpPart<4> w;
        w.c_pix = c_pix; w.c_tdc = c_tdc; w.c_bad = c_bad;
        w.run(p.pk + sp.base, (sp.base & 1) == 0, 0, sp.cnt, p.thr_pix, p.thr_tdc, lane);
        c_pix = w.c_pix; c_tdc = w.c_tdc; c_bad = w.c_bad;
        GAgg a;
        GChain h;
        w.result(&a, &h);
        if (lane == 0) {
            p.ts.agg[tile] = a;
            p.ts.head[tile] = h;
            TileInfo ti;
            ti.first_tdc = w.first_tdc;
            ti.wrap = w.wraps ? 1 : 0;
            p.ts.tinfo[tile] = ti;
        }
    }
    WarpPart<4> w;
    w.c_pix = c_pix; w.c_tdc = c_tdc; w.c_bad = c_bad;
    w.count(p.ctl, lane);
}

// segmented combine: a run start (flag) discards what came before it
struct SAgg { GAgg a; bool f; };
__device__ __forceinline__ SAgg scomb(const SAgg &x, const SAgg &y, long long tp, long long tt) {
    SAgg r;
    r.f = x.f || y.f;
    r.a = y.f ? y.a : acomb(x.a, y.a, tp, tt);
    return r;
}
__device__ __forceinline__ SAgg shfl_up_sagg(const SAgg &v, int o) {
    SAgg u;
    u.a = shfl_up_agg(v.a, o);
    u.f = __shfl_up_sync(0xffffffffu, (int)v.f, o) != 0;
    return u;
}
__device__ __forceinline__ SAgg sid() { SAgg s; s.a = agg_id(); s.f = false; return s; }

// block-wide exclusive segmented scan (SB threads); total in *tot
__device__ SAgg block_excl_sagg(const SAgg &v, SAgg *s_w, SAgg *tot, long long tp, long long tt) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    SAgg incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const SAgg u = shfl_up_sagg(incl, o);
        if (lane >= o) incl = scomb(u, incl, tp, tt);
    }
    SAgg ex = shfl_up_sagg(incl, 1);
    if (lane == 0) ex = sid();
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    if (w == 0) {
        SAgg x = s_w[lane];
        SAgg xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const SAgg u = shfl_up_sagg(xi, o);
            if (lane >= o) xi = scomb(u, xi, tp, tt);
        }
        SAgg xe = shfl_up_sagg(xi, 1);
        if (lane == 0) xe = sid();
        s_w[lane] = xe;
        if (lane == 31) *tot = xi;
    }
    __syncthreads();
    const SAgg r = scomb(s_w[w], ex, tp, tt);
    __syncthreads();
    return r;
}

// a run's first tile restarts the chains (batches only: one stream otherwise)
__device__ __forceinline__ bool run_starts_at(const Params &p, long long tile) {
    return p.bt.tile_run && p.bt.run_tile0[p.bt.tile_run[tile]] == tile;
}

// 32 consecutive stretches of one chain, lane by lane, without a scan of whole
// aggregates: the step into a lane's stretch follows from the last value of the
// nearest lane below that has one, the rest are sums and picks.
struct LaneChain {
    unsigned mask;      // lanes with values
    int step;           // the wrap step into this lane's stretch
    long long prev;     // the last value before it (any_prev: there is one)
    bool any_prev;
    __device__ __forceinline__ void link(const GChain &c, int lane, bool has_in, long long in, long long thr) {
        mask = __ballot_sync(0xffffffffu, c.n > 0);
        const unsigned lower = mask & ((1u << lane) - 1u);
        const long long v = __shfl_sync(0xffffffffu, c.last, lower ? 31 - __clz(lower) : 0);
        any_prev = lower || has_in;
        prev = lower ? v : in;
        step = c.n > 0 && any_prev ? (int)jump(c.first - prev, thr) : 0;
    }
    // lanes below `end` as one stretch
    __device__ __forceinline__ GChain total(const GChain &c, int lane, int end) const {
        const unsigned m = end >= 32 ? mask : mask & ((1u << end) - 1u);
        GChain r;
        r.n = __reduce_add_sync(0xffffffffu, lane < end ? (int)c.n : 0);
        r.sum = __reduce_add_sync(0xffffffffu, lane < end ? (int)c.sum + step : 0);
        r.first = __shfl_sync(0xffffffffu, c.first, m ? __ffs(m) - 1 : 0);
        r.last = __shfl_sync(0xffffffffu, c.last, m ? 31 - __clz(m) : 0);
        return m ? r : chain_id();
    }
};
// one chain's state before each of up to 1024 tiles, a thread per tile, from
// the state E before the first; *step: the wrap step into the tile
struct ScanSm { int n[32], sum[32], has[32]; long long first[32], last[32]; };
__device__ __forceinline__ GChain chain_before(const GChain &c, const GChain &E, ScanSm &S, bool one_warp, long long thr,
                                               int *step) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    bool has_in = E.n > 0;
    long long in = E.last, first = E.n > 0 ? E.first : 0;
    bool has_first = E.n > 0;
    LaneChain l;
    if (!one_warp) {   // the warps before this one: their last value
        const unsigned m = __ballot_sync(0xffffffffu, c.n > 0);
        const long long f = __shfl_sync(0xffffffffu, c.first, m ? __ffs(m) - 1 : 0);
        const long long z = __shfl_sync(0xffffffffu, c.last, m ? 31 - __clz(m) : 0);
        if (lane == 0) {
            S.has[w] = m != 0;
            S.first[w] = f;
            S.last[w] = z;
        }
        __syncthreads();
        const unsigned mw = __ballot_sync(0xffffffffu, lane < w && S.has[lane]);
        if (mw) {
            in = S.last[31 - __clz(mw)];
            has_in = true;
            if (!has_first) first = S.first[__ffs(mw) - 1];
            has_first = true;
        }
    }
    l.link(c, lane, has_in, in, thr);
    int n = (int)c.n, x = (int)c.sum + l.step;
    const int own_n = n, own_x = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, n, o), b = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) { n += a; x += b; }
    }
    int bn = 0, bx = 0;
    if (!one_warp) {
        if (lane == 31) {
            S.n[w] = n;
            S.sum[w] = x;
        }
        __syncthreads();
        bn = __reduce_add_sync(0xffffffffu, lane < w ? S.n[lane] : 0);
        bx = __reduce_add_sync(0xffffffffu, lane < w ? S.sum[lane] : 0);
    }
    const unsigned lower = l.mask & ((1u << lane) - 1u);
    const long long wf = __shfl_sync(0xffffffffu, c.first, l.mask ? __ffs(l.mask) - 1 : 0);
    GChain r;
    r.n = E.n + bn + n - own_n;
    r.sum = E.sum + bx + x - own_x;
    r.last = l.prev;   // E's where nothing lies between
    r.first = has_first ? first : (lower ? wf : 0);
    *step = l.step;
    return r;          // E's wraps count also while there is no value yet
}
// per block of SB tiles: the exclusive scan inside the block (into pre[]) and
// the block's total (into bagg[], its flag into bflag[])
__global__ void __launch_bounds__(SB) k_block_scan(const Params p, GAgg *bagg, int *bflag) {
    __shared__ SAgg s_w[32];
    __shared__ SAgg s_tot;
    const long long t = (long long)blockIdx.x * SB + threadIdx.x;
    SAgg v = sid();
    if (t < p.n_tiles) {
        v.a = p.ts.agg[t];
        v.f = run_starts_at(p, t);
    }
    if (!p.bt.tile_run) {   // one stream: no segments
        __shared__ ScanSm s_scan[2];
        GAgg e;
        int step;
        e.tdc = chain_before(v.a.tdc, chain_id(), s_scan[0], false, p.thr_tdc, &step);
        e.pix = chain_before(v.a.pix, chain_id(), s_scan[1], false, p.thr_pix, &step);
        if (t < p.n_tiles) p.ts.pre[t] = e;
        if (threadIdx.x == SB - 1) {
            bagg[blockIdx.x] = acomb(e, v.a, p.thr_pix, p.thr_tdc);
            bflag[blockIdx.x] = 0;
        }
        return;
    }
    const SAgg ex = block_excl_sagg(v, s_w, &s_tot, p.thr_pix, p.thr_tdc);
    if (t < p.n_tiles) p.ts.pre[t] = v.f ? agg_id() : ex.a;   // a run starts from nothing
    if (threadIdx.x == 0) {
        bagg[blockIdx.x] = s_tot.a;
        bflag[blockIdx.x] = s_tot.f ? 1 : 0;
    }
}

// one block: exclusive segmented scan of the block totals, from the state
// before the call (E0; a batch starts every run from nothing)
__global__ void __launch_bounds__(SB) k_top_scan(const Params p, GAgg *bagg, const int *bflag, long long nb) {
    __shared__ SAgg s_w[32];
    __shared__ SAgg s_tot;
    __shared__ SAgg s_carry;
    const long long tp = p.thr_pix, tt = p.thr_tdc;
    if (!p.bt.tile_run && nb <= 32) {   // one warp does it (up to 1.3e8 packets: 32-bit counts)
        if (threadIdx.x >= 32) return;
        __shared__ ScanSm s_none;
        const long long b = threadIdx.x;
        const GAgg v = b < nb ? bagg[b] : agg_id(), E = p.E0 ? *p.E0 : agg_id();
        GAgg e;
        int step;
        e.tdc = chain_before(v.tdc, E.tdc, s_none, true, tt, &step);
        e.pix = chain_before(v.pix, E.pix, s_none, true, tp, &step);
        if (b < nb) bagg[b] = e;
        return;
    }
    if (threadIdx.x == 0) {
        s_carry.a = (!p.bt.tile_run && p.E0) ? *p.E0 : agg_id();
        s_carry.f = false;
    }
    __syncthreads();
    for (long long b0 = 0; b0 < nb; b0 += SB) {
        const long long b = b0 + threadIdx.x;
        SAgg v = sid();
        if (b < nb) {
            v.a = bagg[b];
            v.f = bflag[b] != 0;
        }
        const SAgg ex = block_excl_sagg(v, s_w, &s_tot, tp, tt);
        const SAgg carry = s_carry;
        const SAgg r = scomb(carry, ex, tp, tt);
        __syncthreads();
        if (b < nb) bagg[b] = r.a;      // now: the state before block b
        if (threadIdx.x == 0) s_carry = scomb(carry, s_tot, tp, tt);
        __syncthreads();
    }
}

// the state before each tile: within its block's scan, after the state before
// the block unless its run started inside the block; the last tile also gives
// the state after the call
__global__ void __launch_bounds__(256) k_apply(const Params p, const GAgg *bpre) {
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
    if (t >= p.n_tiles) return;
    const long long b = t / SB, bstart = b * SB;
    const long long tp = p.thr_pix, tt = p.thr_tdc;
    bool fresh;   // the run of tile t starts inside block b (at or before t)
    if (p.bt.tile_run) fresh = p.bt.run_tile0[p.bt.tile_run[t]] >= bstart;
    else fresh = false;
    const GAgg loc = p.ts.pre[t];
    GAgg e = fresh ? loc : acomb(bpre[b], loc, tp, tt);
    const GAgg g = p.ts.agg[t];
    if (t == p.n_tiles - 1 && !p.bt.tile_run && p.state_out) *p.state_out = acomb(e, g, tp, tt);
    TileInfo ti = p.ts.tinfo[t];
    if (e.pix.n && g.pix.n && jump(g.pix.first - e.pix.last, tp) != 0) {   // the step into the tile's first pixel
        ti.wrap = 1;
        p.ts.tinfo[t] = ti;
    }
    // the range of a tile with triggers before it starts at its first TDC
    // packet: the pixel chain goes on to there
    const long long trig_base = (!p.bt.tile_run && p.E0) ? p.E0->tdc.n : 0;
    if (e.tdc.n > trig_base && ti.first_tdc >= 0) e.pix = ccomb(e.pix, p.ts.head[t], tp);
    p.ts.pre[t] = e;
}

// Up to SB tiles (4 M packets): the whole pre-pass in one launch. A call of a
// few tiles is bound by latency, not by bytes: with a warp per tile the 4096
// packets of a tile are 64 dependent steps of one warp, and three launches
// follow (37 shots, 5 tiles: 30 + 6 + 6 + 4 us; the whole call 112 us, with
// this kernel and two memsets and a copy fewer 69 us; 1000 shots, 117 tiles:
// 125 -> 74 us). Here a CTA takes a tile, its 32 warps two steps each; the
// parts are combined by one warp, from picks and sums (scans of whole aggregates
// took 18 us of 117 tiles, this 14). The CTA that
// finishes last (a counter in the control block) scans the aggregates of all
// tiles and writes the states; nobody waits for anybody.
__device__ __forceinline__ GChain ldcg_chain(const GChain *c) {   // written by another CTA: past L1
    GChain r;
    r.n = __ldcg(&c->n); r.first = __ldcg(&c->first); r.last = __ldcg(&c->last); r.sum = __ldcg(&c->sum);
    return r;
}
template <bool BATCH>
__global__ void __launch_bounds__(SB, 1) k_prepass_small(const Params p, int T) {
    __shared__ GAgg s_a[32];
    __shared__ GChain s_h[32];
    __shared__ int s_first[32];
    __shared__ bool s_wrap[32];
    __shared__ SAgg s_w[32];
    __shared__ SAgg s_tot;
    __shared__ ScanSm s_scan[2];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long tp = p.thr_pix, tt = p.thr_tdc;
    if (blockIdx.x == 0 && threadIdx.x == 0) {   // the fused kernel's last tile writes them
        *p.n_clusters = 0;
        *p.n_trig = 0;
    }
    {
        const long long tile = blockIdx.x;
        const TileSpan sp = tile_span(p, tile, T);
        const int per = T / 32;   // 32, 64 or 128 packets: half a step, one or two
        const int qb = w * per, qe = min(sp.cnt, qb + per);
        WarpPart<2> part;
        if (qb < qe) part.run(p.pk + sp.base, (sp.base & 1) == 0, qb, qe, tp, tt, lane);
        GAgg a;
        GChain h;
        part.result(&a, &h);
        part.count(p.ctl, lane);
        if (lane == 0) {
            s_a[w] = a;
            s_h[w] = h;
            s_first[w] = part.first_tdc;
            s_wrap[w] = part.wraps;
        }
        __syncthreads();
        if (w == 0) {   // the 32 parts in order
            const GAgg mine = s_a[lane];
            LaneChain px, td;
            px.link(mine.pix, lane, false, 0, tp);
            td.link(mine.tdc, lane, false, 0, tt);
            GAgg all;
            all.pix = px.total(mine.pix, lane, 32);
            all.tdc = td.total(mine.tdc, lane, 32);
            const bool wrap = __any_sync(0xffffffffu, px.step != 0 || s_wrap[lane]);
            const unsigned has = __ballot_sync(0xffffffffu, s_first[lane] >= 0);
            const int fl = has ? __ffs(has) - 1 : 0;
            const GChain before = px.total(mine.pix, lane, fl);   // up to the part with the first TDC packet
            if (lane == 0) {
                TileInfo ti;
                ti.first_tdc = has ? s_first[fl] : -1;
                ti.wrap = wrap ? 1 : 0;
                p.ts.tinfo[tile] = ti;
                p.ts.head[tile] = has ? ccomb(before, s_h[fl], tp) : chain_id();
                p.ts.agg[tile] = all;
            }
            __threadfence();
            __syncwarp();
            if (lane == 0) s_last = atomicAdd(&p.ctl->prepass_done, 1u) + 1u == gridDim.x;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the state before every tile (as k_block_scan, k_top_scan and k_apply)
    const long long t = threadIdx.x;
    constexpr bool one = !BATCH;
    const bool one_warp = p.n_tiles <= 32;
    if (one_warp && w > 0) return;
    SAgg v = sid();
    if (t < p.n_tiles) {
        v.a.pix = ldcg_chain(&p.ts.agg[t].pix);
        v.a.tdc = ldcg_chain(&p.ts.agg[t].tdc);
        if constexpr (BATCH) v.f = run_starts_at(p, t);
    }
    GAgg e;
    if constexpr (one) {
        const GAgg E = p.E0 ? *p.E0 : agg_id();
        int step;
        e.tdc = chain_before(v.a.tdc, E.tdc, s_scan[0], one_warp, tt, &step);
        e.pix = chain_before(v.a.pix, E.pix, s_scan[1], one_warp, tp, &step);
    } else {   // a batch: segmented at the runs' first tiles
        SAgg ex;
        if (one_warp) {
            SAgg incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const SAgg u = shfl_up_sagg(incl, o);
                if (lane >= o) incl = scomb(u, incl, tp, tt);
            }
            ex = shfl_up_sagg(incl, 1);
            if (lane == 0) ex = sid();
        } else {
            ex = block_excl_sagg(v, s_w, &s_tot, tp, tt);
        }
        e = v.f ? agg_id() : ex.a;
    }
    if (t >= p.n_tiles) return;
    if (t == p.n_tiles - 1 && one && p.state_out) *p.state_out = acomb(e, v.a, tp, tt);
    TileInfo ti;
    ti.first_tdc = __ldcg(&p.ts.tinfo[t].first_tdc);
    ti.wrap = __ldcg(&p.ts.tinfo[t].wrap);
    if (e.pix.n && v.a.pix.n && jump(v.a.pix.first - e.pix.last, tp) != 0) {   // the step into the tile's first pixel
        ti.wrap = 1;
        p.ts.tinfo[t] = ti;
    }
    const long long trig_base = (one && p.E0) ? p.E0->tdc.n : 0;
    if (e.tdc.n > trig_base && ti.first_tdc >= 0) {
        e.pix = ccomb(e.pix, ldcg_chain(p.ts.head + t), tp);
    }
    p.ts.pre[t] = e;
}

}  // namespace

size_t unwrap_prepass_scratch_bytes(long long n_tiles) {
    const long long nb = (n_tiles + SB - 1) / SB + 1;
    return (size_t)nb * (sizeof(GAgg) + sizeof(int)) + 256;
}

cudaError_t launch_unwrap_prepass(const Params &p, int T, int grid, cudaStream_t s) {
    if (p.n_tiles <= 0) return cudaSuccess;
    if (p.n_tiles <= SB) {
        if (p.bt.tile_run) k_prepass_small<true><<<(unsigned)p.n_tiles, SB, 0, s>>>(p, T);
        else k_prepass_small<false><<<(unsigned)p.n_tiles, SB, 0, s>>>(p, T);
        return cudaGetLastError();
    }
    const long long nb = (p.n_tiles + SB - 1) / SB;
    GAgg *bagg = p.ts.blk;
    int *bflag = reinterpret_cast<int *>(bagg + nb + 1);
    long long g = (p.n_tiles + AW - 1) / AW;
    if (g > (long long)grid * 8) g = (long long)grid * 8;
    k_tile_aggs<<<(unsigned)g, AW * 32, 0, s>>>(p, T);
    k_block_scan<<<(unsigned)nb, SB, 0, s>>>(p, bagg, bflag);
    k_top_scan<<<1, SB, 0, s>>>(p, bagg, bflag, nb);
    k_apply<<<(unsigned)((p.n_tiles + 255) / 256), 256, 0, s>>>(p, bagg);
    return cudaGetLastError();
}

}  // namespace tpxk
