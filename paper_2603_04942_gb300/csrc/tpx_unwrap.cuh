// tpx_unwrap.cuh -- a warp's pass over a stretch of packets: the aggregates of
// both unwrap chains (Sec. IV.A), for the fused kernel's pre-pass and for the
// general path's decode.
#pragma once

#include <cstdint>

#include "tpx_common.cuh"
#include "tpx_fused.cuh"

namespace tpxk {

// Stream-order accumulation of one chain by a warp, 64 packets per step (two
// per lane). Per lane: its pair's first / last raw value and the wrap steps
// inside the pair; across lanes: the last value of the nearest lower lane
// that has one (ballot), and the last value of the previous step.
struct WarpChain {
    long long first, last, sum;   // sum: per lane, of the steps it detected
    long long n;
    bool any;
};
// Returns whether this lane found a wrap step.
__device__ __forceinline__ bool warp_chain_step(WarpChain &c, bool h0, long long r0, bool h1, long long r1,
                                                long long thr, int lane) {
    const bool has = h0 || h1;
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (!m) return false;
    const long long pf = h0 ? r0 : r1;       // first of the pair
    const long long pl = h1 ? r1 : r0;       // last of the pair
    long long s = (h0 && h1) ? jump(r1 - r0, thr) : 0;
    bool found = s != 0;
    // the value before this pair: the last one of the nearest lower lane with
    // a value, else the chain's last value before this step
    const unsigned lower = m & ((1u << lane) - 1u);
    const int src = lower ? 31 - __clz(lower) : 0;
    const long long prev_lane = __shfl_sync(0xffffffffu, pl, src);
    if (has && (lower || c.any)) {
        const long long b = jump(pf - (lower ? prev_lane : c.last), thr);
        s += b;
        found |= b != 0;
    }
    c.sum += s;
    const int lo = __ffs(m) - 1, hi = 31 - __clz(m);
    const long long step_first = __shfl_sync(0xffffffffu, pf, lo);
    const long long step_last = __shfl_sync(0xffffffffu, pl, hi);
    if (!c.any) c.first = step_first;
    c.last = step_last;
    c.any = true;
    c.n += __popc(m) + __popc(__ballot_sync(0xffffffffu, h0 && h1));
    return found;
}

// Bound by the packet stream's bytes once the loads run ahead: KS steps of 64
// packets are in flight per warp while the previous KS are combined. A step of
// pixels only (the common one) takes a short path: the neighbour lane's last
// value by one shuffle, the wrap test on both differences, nothing to rank.
template <int KS>
struct WarpPart {
    WarpChain cp{0, 0, 0, 0, false}, ct{0, 0, 0, 0, false}, ch{0, 0, 0, 0, false};
    int first_tdc = -1;
    bool wraps = false;       // this lane (after result(): some lane) saw a pixel wrap step
    bool tdc_wraps = false;   // this lane saw a TDC wrap step
    unsigned long long c_pix = 0, c_tdc = 0, c_bad = 0;   // of this lane

    // packets [qb, qe) of the tile at src (qb even); vec: src is 16-byte aligned
    __device__ __forceinline__ void run(const uint64_t *src, bool vec, int qb, int qe, long long tp, long long tt, int lane) {
        // the lane's two packets of each step from q0 on (zero past the end)
        auto load = [&](int q0, uint64_t (&v)[2 * KS]) {
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                const int q = q0 + 64 * k + 2 * lane;
                uint64_t a = 0, b = 0;
                if (vec && q + 1 < qe) {
                    const ulonglong2 u = __ldcs(reinterpret_cast<const ulonglong2 *>(src + q));
                    a = u.x;
                    b = u.y;
                } else {
                    if (q < qe) a = __ldcs(src + q);
                    if (q + 1 < qe) b = __ldcs(src + q + 1);
                }
                v[2 * k] = a;
                v[2 * k + 1] = b;
            }
        };
        auto step = [&](int q0, uint64_t w0, uint64_t w1) {
            const int q = q0 + 2 * lane;
            const unsigned h0 = (unsigned)(w0 >> 60), h1 = (unsigned)(w1 >> 60);
            const bool p0 = h0 == 0xBu, p1 = h1 == 0xBu;   // zero past the end: neither
            if (__all_sync(0xffffffffu, p0 && p1)) {
                const long long r0 = pix_raw(w0), r1 = pix_raw(w1);
                long long prev = __shfl_up_sync(0xffffffffu, r1, 1);
                if (lane == 0) prev = cp.any ? cp.last : r0;
                const long long s = jump(r1 - r0, tp) + jump(r0 - prev, tp);
                wraps |= jump(r1 - r0, tp) != 0 || jump(r0 - prev, tp) != 0;
                cp.sum += s;
                if (!cp.any) cp.first = __shfl_sync(0xffffffffu, r0, 0);
                cp.last = __shfl_sync(0xffffffffu, r1, 31);
                cp.any = true;
                cp.n += 64;
                c_pix += 2;
                return;
            }
            const bool in0 = q < qe, in1 = q + 1 < qe;
            const bool t0 = in0 && h0 == 0x6u, t1 = in1 && h1 == 0x6u;
            c_pix += (unsigned)p0 + (unsigned)p1;
            c_tdc += (unsigned)t0 + (unsigned)t1;
            c_bad += (unsigned)(in0 && !p0 && !t0) + (unsigned)(in1 && !p1 && !t1);
            const long long r0 = p0 ? pix_raw(w0) : 0, r1 = p1 ? pix_raw(w1) : 0;
            const unsigned mt = __ballot_sync(0xffffffffu, t0 || t1);
            if (mt && first_tdc < 0) {   // the pixel chain up to the first TDC packet
                const int fl = __ffs(mt) - 1;
                first_tdc = __shfl_sync(0xffffffffu, t0 ? q : q + 1, fl);
                ch = cp;
                warp_chain_step(ch, p0 && q < first_tdc, r0, p1 && q + 1 < first_tdc, r1, tp, lane);
            }
            wraps |= warp_chain_step(cp, p0, r0, p1, r1, tp, lane);
            if (mt) tdc_wraps |= warp_chain_step(ct, t0, t0 ? tdc_raw(w0) : 0, t1, t1 ? tdc_raw(w1) : 0, tt, lane);
        };
        uint64_t cur[2 * KS], nxt[2 * KS];
        load(qb, nxt);
        for (int q0 = qb; q0 < qe; q0 += 64 * KS) {
#pragma unroll
            for (int k = 0; k < 2 * KS; ++k) cur[k] = nxt[k];
            if (q0 + 64 * KS < qe) load(q0 + 64 * KS, nxt);
#pragma unroll
            for (int k = 0; k < KS; ++k)
                if (q0 + 64 * k < qe) step(q0 + 64 * k, cur[2 * k], cur[2 * k + 1]);
        }
    }
    // the part's aggregates, the same in every lane: both chains, and the pixel
    // chain up to the first TDC packet; wraps: whether a pixel wrap lies inside
    __device__ __forceinline__ void result(GAgg *a, GChain *h) {
        long long sp_ = cp.sum, st_ = ct.sum, sh_ = ch.sum;
        wraps = __any_sync(0xffffffffu, wraps);
        if (wraps || __any_sync(0xffffffffu, st_ != 0)) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sp_ += __shfl_xor_sync(0xffffffffu, sp_, o);
                st_ += __shfl_xor_sync(0xffffffffu, st_, o);
                sh_ += __shfl_xor_sync(0xffffffffu, sh_, o);
            }
        }
        a->pix.n = cp.n; a->pix.first = cp.first; a->pix.last = cp.last; a->pix.sum = sp_;
        a->tdc.n = ct.n; a->tdc.first = ct.first; a->tdc.last = ct.last; a->tdc.sum = st_;
        if (!cp.any) a->pix = chain_id();
        if (!ct.any) a->tdc = chain_id();
        h->n = ch.n; h->first = ch.first; h->last = ch.last; h->sum = sh_;
        if (!ch.any) *h = chain_id();
    }
    // packet-class counters of the call (Ctl is cleared before the launch)
    __device__ __forceinline__ void count(Ctl *ctl, int lane) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c_pix += __shfl_xor_sync(0xffffffffu, c_pix, o);
            c_tdc += __shfl_xor_sync(0xffffffffu, c_tdc, o);
            c_bad += __shfl_xor_sync(0xffffffffu, c_bad, o);
        }
        if (lane == 0) {
            if (c_pix) atomicAdd(&ctl->counters[C_PIXELS], c_pix);
            if (c_tdc) atomicAdd(&ctl->counters[C_TDCS], c_tdc);
            if (c_bad) atomicAdd(&ctl->counters[C_CORRUPT], c_bad);
        }
    }
};

}  // namespace tpxk
