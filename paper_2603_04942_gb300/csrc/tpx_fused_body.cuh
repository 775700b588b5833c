// tpx_fused_body.cuh -- the fused kernel, included once per tile geometry
// by tpx_fused.cu inside a namespace that defines NT (threads per CTA),
// T (packets per tile), C (range capacity), TR (rows of the cell table), MS
// (trigger packets a range may hold), MINB (CTAs per SM) and BIG_REGION (bytes
// of shared scratch of the big-range path). No include guard: it
// is meant to be included repeatedly.
//
// Bound by instruction issue and by the barriers between its phases, not by
// bytes (18 B per packet, 5% of the copy bandwidth). Measured on 2.46e8 packets
// of the large recipe, 2048-packet tiles: 61.9 -> 41.7 us per 10^6 packets,
// 45.4 -> 29.8 warp instructions per packet, against the form with a chained
// hash of the pixels in arrival order, a walk for the unwrap chains and the
// copy-out as a phase of the workers.
//
// A CTA is NW worker warps, which cluster one tile's range after the other,
// and one service warp, which claims and plans the next tile and copies the
// finished tiles' records out meanwhile. The workers synchronise among
// themselves (cta_sync); the two sides hand tiles over through counters in
// shared memory.
constexpr int NW = NT / 32 - 1;    // worker warps
constexpr int NTW = 32 * NW;       // worker threads
constexpr int MAXSEG = MS;         // TDC packets a range may hold (more: the call is redone)
constexpr uint64_t INVALID = ~0ull;
constexpr uint32_t EMPTY = 0xFFFFu;
constexpr long long MAX_SPIN = 1LL << 22;   // bounded look-back waits (~0.5 s)
constexpr long long MAX_TRIES = 1LL << 18;  // bounded look-back waits of the service warp (~0.5 s)
constexpr long long MAX_HANDOVER = 1LL << 25;   // bounded waits between the two sides (seconds)

static_assert(T <= C && C % 1024 == 0, "tile geometry");
constexpr int LOOK = C / T > 4 ? C / T : 4;   // tiles after its own that a range within the capacity can reach into
static_assert(C % T == 0 || LOOK * T >= C, "tiles of a range");
constexpr int KM = (C + NTW - 1) / NTW;   // packets of a range a worker thread holds
constexpr int TB = 256 * TR;              // cell table: bits, words
constexpr int TW = TB / 32;
constexpr int OHB = C >= 8192 ? 2048 : 1024;   // buckets of the second hits of a table cell
constexpr uint16_t NOLAB = 0xFFFFu, PEAK = 0x4000u;   // a position's label entry
constexpr int QN = C / 2;          // pairs the union queue holds
static_assert(C <= 0x4000 && (TR & (TR - 1)) == 0 && TR >= 256, "16-bit slots, positions and label entries");
__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NTW) : "memory"); }

// ------------------------------------------------------------------ helpers
// Checked build (-DTPX_CHECKED): every data-dependent shared-memory or global
// index (hash chains, member lists, roots, cluster ids, output positions) is
// tested against its array before use; a violation sets ST_BOUNDS in the
// status word and skips the access. The normal build compiles the tests away.
#ifdef TPX_CHECKED
__device__ __forceinline__ bool in_bounds(long long i, long long n, const Params &p) {
    if (i >= 0 && i < n) return true;
    atomicOr(&p.ctl->status, ST_BOUNDS);
    return false;
}
#define TPX_IN(i, n) in_bounds((long long)(i), (long long)(n), p)
#else
#define TPX_IN(i, n) true
#endif

// Phase timing (-DTPX_PHASE_TIMING, the libtpx_phases.so build): lane 0 of
// every warp adds the clock64 cycles since the previous mark to the phase's
// counter; the kernel's end adds the CTA's counters to g_phase. A phase's
// time includes the barrier wait that ends it. The normal build compiles the
// marks away.
#ifdef TPX_PHASE_TIMING
__device__ unsigned long long g_phase[32];
#define TPX_PH(k)                                                                         \
    do {                                                                                  \
        const long long ph_now = clock64();                                               \
        if ((threadIdx.x & 31) == 0) atomicAdd(&S.ph[k], (unsigned long long)(ph_now - ph_t)); \
        ph_t = ph_now;                                                                    \
    } while (0)
#else
#define TPX_PH(k) do {} while (0)
#endif

// kept-pixel record: [63:40] tof+bias | [39:30] ToT | [29:16] segment | [15:8] y | [7:0] x;
// the low 30 bits are the pixel's cell (segment, y, x)
__device__ __forceinline__ uint64_t mkrec(uint32_t tofb, uint32_t seg, uint32_t tot, uint32_t x, uint32_t y) {
    return ((uint64_t)tofb << 40) | ((uint64_t)tot << 30) | ((uint64_t)seg << 16) | ((uint64_t)y << 8) | x;
}
__device__ __forceinline__ int r_x(uint64_t r) { return (int)(r & 255); }
__device__ __forceinline__ int r_y(uint64_t r) { return (int)((r >> 8) & 255); }
__device__ __forceinline__ int r_seg(uint64_t r) { return (int)((r >> 16) & 0x3FFF); }
__device__ __forceinline__ int r_tot(uint64_t r) { return (int)((r >> 30) & 1023); }
__device__ __forceinline__ int r_tof(uint64_t r) { return (int)(r >> 40); }
__device__ __forceinline__ uint32_t r_cell(uint64_t r) { return (uint32_t)r & 0x3FFFFFFFu; }
// |d| <= dt, for 0 <= dt < 2^31
__device__ __forceinline__ bool within(int d, int dt) { return (uint32_t)d + (uint32_t)dt <= 2u * (uint32_t)dt; }

// The flags are polled with relaxed loads and a fence follows once they are
// all there: an acquiring load empties the SM's L1, which the CTA's big-range
// path reads through, at every poll (2.4x the time of an uneven batch).
__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A (segment, y, x) cell's bit of the cell table: TR rows of 256 columns, the
// rows of a shot shifted by its number, so that a row of cells is a run of bits
// and the row above it the run 256 bits on. The kept pixels that find their
// bit free take slots in the order of the bits (the table with the rank of
// each word), so a pixel's right-hand neighbour is the next slot and the
// neighbours in a row consecutive slots; a pixel that finds its bit taken (a
// second hit of the cell, or another shot's cell) takes a slot after all of
// them and a place in a chained hash.
constexpr uint32_t HS = 101u << 8;
__device__ __forceinline__ uint32_t tbit(uint64_t r) {
    return (((uint32_t)r & 0xFFFFu) + HS * (uint32_t)r_seg(r)) & (TB - 1);
}
__device__ __forceinline__ uint32_t ohash(uint32_t bit) { return (bit ^ (bit >> 9)) & (OHB - 1); }

// Union-find over 16-bit parents addressed in the shared window (pb: the
// array's shared address). Pointers set by the neighbour pass go forward in
// (y, x); roots are linked the larger slot under the smaller.
__device__ __forceinline__ uint32_t uf_ld(uint32_t pb, uint32_t x) {
    unsigned short v;
    asm volatile("ld.volatile.shared.u16 %0, [%1];" : "=h"(v) : "r"(pb + 2 * x) : "memory");
    return v;
}
__device__ __forceinline__ void uf_st(uint32_t pb, uint32_t x, uint32_t v) {
    asm volatile("st.volatile.shared.u16 [%0], %1;" ::"r"(pb + 2 * x), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ uint32_t uf_cas(uint32_t pb, uint32_t x, uint32_t cmp, uint32_t v) {
    unsigned short o;
    asm volatile("atom.shared.cas.b16 %0, [%1], %2, %3;"
                 : "=h"(o) : "r"(pb + 2 * x), "h"((unsigned short)cmp), "h"((unsigned short)v) : "memory");
    return o;
}
__device__ __forceinline__ uint32_t uf_find(uint32_t pb, uint32_t x) {
    for (;;) {
        const uint32_t px = uf_ld(pb, x);
        if (px == x) return x;
        const uint32_t g = uf_ld(pb, px);
        if (g == px) return px;
        uf_st(pb, x, g);   // path halving: g is an ancestor of x
        x = g;
    }
}
__device__ __forceinline__ uint32_t uf_root(uint32_t pb, uint32_t x) {   // changes nothing
    uint32_t px;
    while ((px = uf_ld(pb, x)) != x) x = px;
    return x;
}
// lock-free union: the larger root slot is linked under the smaller
__device__ void uf_unite(uint32_t pb, uint32_t a, uint32_t b) {
    for (;;) {
        a = uf_find(pb, a);
        b = uf_find(pb, b);
        if (a == b) return;
        const uint32_t lo = min(a, b), hi = max(a, b);
        if (uf_cas(pb, hi, hi, lo) == hi) return;
        a = lo;
        b = hi;   // hi was linked meanwhile: find again
    }
}

// --------------------------------------------------------------- smem layout
struct __align__(16) Smem {
    union {
        struct {
            uint64_t srec[C + 4];     // while the range is read: its TDC packets (all packets
                                      // where a pixel wrap is near) by position; then the
                                      // kept-pixel records by slot
            uint16_t spos[C];         // wraps by position where a wrap is near; then the
                                      // records' positions in the range
            uint16_t par[C];          // union-find parents, then roots
            union {
                struct { uint32_t bits[TW]; uint16_t rank[TW], ohead[OHB]; } t;
                uint32_t mhead[C];
            } u1;                     // the cell table, then (CC) member-list heads and labels by root
            union { uint32_t queue[QN]; uint16_t mnext[C]; uint16_t lab[C]; } u2;
                                      // pairs left to unite, member links, labels by position
            union { uint16_t onext[C]; uint16_t rootpos[C]; } u5;   // chains of second hits; CC: the roots
            uint8_t notpeak[C];
            union { uint32_t lbits[C / 32]; uint32_t tmask[C / 32]; uint32_t rwalk[C / 32]; } u3;
                                      // TDC packets of each 32 positions; slots to walk again;
                                      // then the label positions, one bit each
            union { uint16_t lpre[C / 32]; uint16_t tpre[C / 32]; } u4;   // bits before each word
        };
        unsigned char big[BIG_REGION];   // the big-range path's shared scratch
    };
    long long tdc_t[MAXSEG + 1];  // unwrapped trigger times of the range, and a time past all
    uint16_t tdc_pos[MAXSEG];     // their positions
    // the tile in work and the next one, planned by the service warp
    struct Plan {
        GAgg E;                   // unwrap state before the range (pixels) and the tile (TDCs)
        long long tile;
        int f, w0, len, term, slow;
        unsigned status;
    } plan[2];
    long long j0;                 // pixel wrap step from the last pixel before the range to its first
    int warp_int[NW + 2];
    unsigned long long cnt[C_NUM];   // this tile's counters
    unsigned long long acc[C_NUM];   // this CTA's counters, added to the call's at its end
    long long clo;                // unstaged: the tile's record offset
    // finished tiles awaiting their offsets: entry k of the CTA, staged in slot
    // k % (1 for a single stream, RING in a batch). A tile with nothing to write
    // (most tiles of a run whose shots span several) takes none.
    struct Pend {
        long long tile, ntr;      // the tile; its trigger total (single streams)
        long long at;             // STAGED_ONLY: where its records are staged
        int ncl, ntdc, run;       // its records and triggers; its run
        bool first, big;          // the run's first tile; records in the big-range slot
    } pend[4];
    // the handover: tiles planned and finished, entries made and copied out
    // (monotonic counts)
    int planned, produced, entries, consumed;
    int first_pix;                // first pixel of the range
    int ntdc;                     // TDC packets of the range
    int nroot;                    // clusters of the tile
    int nov;                      // kept pixels that found their table bit taken
    int qn, rw;                   // pairs queued for a union; a slot has to be walked again
    unsigned n_pre, n_bg, n_pk;   // dropped before a trigger, background, local maxima
    unsigned status;
#ifdef TPX_PHASE_TIMING
    unsigned long long ph[32];
#endif
};

// MINB CTAs per SM within the SM's 228 KB of shared memory (1 KB of it is
// reserved per CTA)
static_assert(MINB * (sizeof(Smem) + 1024) <= 228 * 1024, "shared memory of the tile geometry");

// a batch keeps up to RING finished tiles per CTA waiting for their offsets (a
// tile behind a big range need not wait for it); a single stream keeps one
constexpr int RING = kBatchRing;
static_assert(RING >= 1 && RING <= 4, "the ring of staged tiles");

// ---------------------------------------------------- big-range constants
// (the path itself is described at big_range below)
constexpr int BR_L = 65535;          // positions of a big range (16-bit)
constexpr int BR_LW = (BR_L + 1) / 32;
constexpr int BR_S = 256;            // shots (trigger packets) of a big range
// sort keys (time bin, x stripe) shared out over its shots
constexpr int BR_BINS = C >= 8192 ? 12288 : 4096;
constexpr int BR_NS = 32;            // x stripes of 8 columns (16 when rx > 8, one when rx > 16)
struct BrMom { unsigned long long s_tot, s_x, s_y, s_tt, best; unsigned n, npk; };
static_assert(sizeof(BrMom) == 48, "moment record");
// shared scratch: the tile arrays in front of the trigger tables
constexpr int BR_REGION = (int)offsetof(Smem, tdc_t);
static_assert(BR_REGION >= BIG_REGION, "the big-range scratch");
// the neighbour pass chains the pixels by cell: heads in place of the sort's
// bins, and the chains of the first BR_NX pixels in shared memory (the others'
// in the scratch); the window pass reads the sorted records through the same
// place, BR_CH pixels at a time with those before them
constexpr int BR_NX = 16 * NT;
constexpr int BR_CH = 2 * NT, BR_SB = 4 * NT;
static_assert(8 * BR_SB <= 2 * BR_NX, "the window's records in the chains' place");
constexpr int BR_FIXED = 4 * (BR_BINS + 4) + 4 * BR_LW + 2 * BR_LW + 4 * 5 * BR_S + 4 * 16 + 2 * BR_NX;
// kept pixels: a 16-bit parent and a local-maximum bit each
constexpr int BR_N0 = ((BR_REGION - BR_FIXED) * 8 / 17) & ~63;
constexpr int BR_N = BR_N0 < 65472 ? BR_N0 : 65472;
static_assert(BR_N > C && BR_N % 64 == 0, "a big range holds more pixels than a tile");
static_assert(2 * BR_N + BR_N / 8 + BR_FIXED <= BR_REGION, "big-range shared scratch");
// per-CTA global scratch: records by position, sorted records and their
// positions, moments by root, and the staged cluster records (a big range
// may hold up to one cluster per kept pixel)
constexpr size_t BR_REC_OFF = ((size_t)8 * (BR_L + 1) + (size_t)58 * BR_N + 255) & ~(size_t)255;
// One record slot per ring entry: a big range's records wait in its entry's
// slot while the CTA goes on.
constexpr size_t BR_STRIDE = (BR_REC_OFF + RING * sizeof(tpx_record) * (size_t)BR_N + 255) & ~(size_t)255;
__device__ __forceinline__ tpx_record *br_stage(const Params &p, int slot) {
    return reinterpret_cast<tpx_record *>(p.big + (size_t)blockIdx.x * BR_STRIDE + BR_REC_OFF) + (size_t)slot * BR_N;
}


// block exclusive scan in thread order of two 16-bit halves added
// separately (__vadd2); each half's sums must fit it. Total in *total.
__device__ unsigned block_scan_vadd2(Smem &S, unsigned v, unsigned *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl = __vadd2(incl, u);
    }
    if (lane == 31) S.warp_int[w] = (int)incl;
    cta_sync();
    if (w == 0) {
        const unsigned x = lane < NW ? (unsigned)S.warp_int[lane] : 0u;
        unsigned xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi = __vadd2(xi, u);
        }
        if (lane < NW) S.warp_int[lane] = (int)__vsub2(xi, x);
        if (lane == NW - 1) S.warp_int[NW] = (int)xi;
    }
    cta_sync();
    const unsigned r = __vadd2((unsigned)S.warp_int[w], __vsub2(incl, v));
    *total = (unsigned)S.warp_int[NW];
    cta_sync();
    return r;
}

// block exclusive scan of int; total in *total
__device__ int block_scan_int(Smem &S, int v, int *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) S.warp_int[w] = incl;
    cta_sync();
    if (w == 0) {
        int x = lane < NW ? S.warp_int[lane] : 0;
        int xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += u;
        }
        if (lane < NW) S.warp_int[lane] = xi - x;
        if (lane == NW - 1) S.warp_int[NW] = xi;
    }
    cta_sync();
    int r = S.warp_int[w] + incl - v;
    *total = S.warp_int[NW];
    cta_sync();
    return r;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// once any wait has run out, every later wait gives up at once, so a broken
// chain costs one bounded wait, not one per tile
__device__ __forceinline__ bool timed_out(const Params &p) {
    return (*reinterpret_cast<volatile unsigned *>(&p.ctl->status) & ST_DEVTIMEOUT) != 0;
}

// Bounded decoupled look-back, one warp. Each trip reads the flags of
// 32 * LB predecessors at once (lane l holds tiles hi - LB*l - j, j = 0 the
// latest), waits only for the tiles from hi down to the nearest inclusive
// prefix, and combines them in stream order. Two dependent L2 round trips
// per trip (flags, then values), so wide trips keep the chain short.
constexpr int LBC = 4;

// per lane: which of its LB tiles are needed this trip, given the flags
struct LbScan { unsigned need, inc; int stop; bool ok; };
template <int LB>
__device__ __forceinline__ LbScan lb_scan(const unsigned *flags, long long hi, long long lo, unsigned seq) {
    const int lane = threadIdx.x & 31;
    unsigned rdy = 0, inc = 0;
#pragma unroll
    for (int j = 0; j < LB; ++j) {
        const long long q = hi - LB * lane - j;
        if (q < lo) { rdy |= 1u << j; continue; }
        const unsigned f = ld_relaxed(&flags[q]);
        if ((f >> 2) == seq && (f & 3u)) {
            rdy |= 1u << j;
            if ((f & 3u) == 2u) inc |= 1u << j;
        }
    }
    const unsigned im = __ballot_sync(0xffffffffu, inc != 0);
    LbScan r;
    r.stop = im ? __ffs(im) - 1 : 31;
    r.inc = inc;
    const unsigned all = (1u << LB) - 1u;
    r.need = lane < r.stop ? all : (lane == r.stop ? (inc ? ((inc & (0u - inc)) << 1) - 1u : all) : 0u);
    r.ok = (rdy & r.need) == r.need;
    return r;
}

// Decoupled look-back over the record counts of the tiles (and, in a batch,
// their trigger counts: .y), over all tiles of the call.
template <bool BATCH>
__device__ longlong2 lookback_count_warp(const Params &p, long long tile, unsigned seq, unsigned *status,
                                         bool block = true, bool *ready = nullptr) {
    const int lane = threadIdx.x & 31;
    longlong2 acc = make_longlong2(0, 0);
    for (long long hi = tile - 1; hi >= 0; hi -= 32 * LBC) {
        LbScan sc;
        long long spins = 0;
        for (;;) {
            sc = lb_scan<LBC>(p.ts.cflags, hi, 0, seq);
            if (__all_sync(0xffffffffu, sc.ok)) break;
            if (!block) { *ready = false; return acc; }   // not yet: the caller tries again later
            if (++spins > MAX_SPIN || timed_out(p)) {
                if (lane == 0) atomicOr(&p.ctl->status, ST_DEVTIMEOUT);
                *status |= ST_DEVTIMEOUT;
                return acc;
            }
            __nanosleep(64);
        }
        __threadfence();
        long long v = 0, w = 0;
#pragma unroll
        for (int j = 0; j < LBC; ++j) {
            const long long q = hi - LBC * lane - j;
            if (q < 0 || !((sc.need >> j) & 1u)) continue;
            const bool inc = (sc.inc >> j) & 1u;
            v += __ldcg(inc ? &p.ts.cpre[q] : &p.ts.cagg[q]);
            if (BATCH) w += __ldcg(inc ? &p.bt.tcpre[q] : &p.bt.tcagg[q]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, o);
            if (BATCH) w += __shfl_xor_sync(0xffffffffu, w, o);
        }
        acc.x += v;
        acc.y += w;
        if (__any_sync(0xffffffffu, sc.inc != 0)) break;
    }
    return acc;
}

static_assert((C / 32) % 32 == 0, "the position bitmaps split evenly over a warp");

// the slot of the table's first pixel at or after a bit
__device__ __forceinline__ int rank_at(const Smem &S, uint32_t bit) {
    return (int)S.u1.t.rank[bit >> 5] + __popc(S.u1.t.bits[bit >> 5] & ((1u << (bit & 31)) - 1u));
}
// the slots [*s0, *s1) of the table's pixels in the cells dlo..dhi columns from
// the cell at `bit` (of column x), in the row dy above
__device__ __forceinline__ void row_slots(const Smem &S, uint32_t bit, int dy, int dlo, int dhi, int *s0, int *s1) {
    const uint32_t row = (bit + 256u * (uint32_t)dy) & (TB - 1);
    *s0 = rank_at(S, row + dlo);
    const uint32_t e = row + dhi;
    *s1 = rank_at(S, e) + (int)((S.u1.t.bits[e >> 5] >> (e & 31)) & 1u);
}

// The columns dlo..dhi from bit `row` of a table row that can hold pixels outside
// the table: those found their cell's bit taken. (In a narrow row nearly all are.)
__device__ __forceinline__ uint32_t taken_columns(const Smem &S, uint32_t row, int dlo, int dhi) {
    uint32_t m = (2u << (dhi - dlo)) - 1u;
    if (dhi - dlo > 4) {
        const uint32_t at = row + (uint32_t)dlo, k = at >> 5;
        m &= __funnelshift_r(S.u1.t.bits[k], S.u1.t.bits[min(k + 1, (uint32_t)TW - 1)], at & 31u);
    }
    return m;
}

// Walks a table pixel's candidates again and unites it with each partner in
// the forward half of its box (Sec. V.A).
__device__ void rewalk_unite(const Smem &S, const Params &p, uint32_t pb, int i) {
    const uint64_t r = S.srec[i];
    const int x = r_x(r), y = r_y(r), tb = r_tof(r);
    const uint32_t bit = tbit(r), cell = r_cell(r);
    for (int dy = 0; dy <= p.ry && y + dy <= 255; ++dy) {
        const int dlo = dy == 0 ? 0 : -min(p.rx, x), dhi = min(p.rx, 255 - x);
        int j, s1;
        row_slots(S, bit, dy, dlo, dhi, &j, &s1);
        for (; j < s1; ++j) {
            if (j == i || !TPX_IN(j, C)) continue;
            const uint64_t rj = S.srec[j];
            if (r_cell(rj) - (cell + (uint32_t)(256 * dy + dlo)) > (uint32_t)(dhi - dlo)) continue;
            if (within(r_tof(rj) - tb, p.dt)) uf_unite(pb, (uint32_t)i, (uint32_t)j);
        }
    }
}

// An adjacent pair's local-maximum flags: equal ToT goes to the later pixel
// (Sec. V.B).
__device__ __forceinline__ bool dimmer(const Smem &S, int i, int tot, int j, int aj) {
    return aj > tot || (aj == tot && S.spos[j] > S.spos[i]);
}

// A pair left to unite once the pointers stand; a full queue marks the pixel
// for a second walk.
__device__ __forceinline__ void queue_pair(Smem &S, int i, int j) {
    const int at = atomicAdd(&S.qn, 1);
    if (at < QN) S.u2.queue[at] = ((uint32_t)i << 16) | (uint32_t)j;
    else { atomicOr(&S.u3.rwalk[i >> 5], 1u << (i & 31)); S.rw = 1; }
}

// One row (dy above) of the box of a pixel outside the table: its adjacent
// pixels in the table, and among the others those after it.
// CC: the pairs are queued, or united at once in a second walk.
template <int MODE, bool UNITE>
__device__ __forceinline__ void overflow_row_in(Smem &S, const Params &p, uint32_t pb, int o, int dy, int nb) {
    const int i = nb + o;
    const uint64_t r = S.srec[i];
    const int x = r_x(r), y = r_y(r), tb = r_tof(r), tot = r_tot(r);
    if (y + dy < 0 || y + dy > 255) return;
    const uint32_t bit = tbit(r), cell = r_cell(r);
    const int dlo = -min(p.rx, x), dhi = min(p.rx, 255 - x);
    const uint32_t c0 = cell + (uint32_t)(256 * dy + dlo);
    auto visit = [&](int j) {
        const uint64_t rj = S.srec[j];
        if (r_cell(rj) - c0 > (uint32_t)(dhi - dlo) || !within(r_tof(rj) - tb, p.dt)) return;
        S.notpeak[dimmer(S, i, tot, j, r_tot(rj)) ? i : j] = 1;
        if (MODE != TPX_MODE_CC) return;
        if (UNITE) uf_unite(pb, (uint32_t)i, (uint32_t)j); else queue_pair(S, i, j);
    };
    int j, s1;
    row_slots(S, bit, dy, dlo, dhi, &j, &s1);
    for (; j < s1; ++j)
        if (TPX_IN(j, C)) visit(j);
    const uint32_t row = (bit + 256u * (uint32_t)dy) & (TB - 1);
    for (uint32_t m = taken_columns(S, row, dlo, dhi); m; m &= m - 1) {
        const int d = __ffs(m) - 1;
        for (uint32_t q = S.u1.t.ohead[ohash(row + dlo + d)]; q != EMPTY; q = S.u5.onext[q]) {
            if (!TPX_IN(nb + q, C)) break;
            // (cells of the same chain: visited for the cell they are in)
            if ((int)q > o && r_cell(S.srec[nb + q]) == c0 + d) visit(nb + (int)q);
        }
    }
}

// Few pixels come here, so in CC mode it is a call (600,000 shots 33.49 -> 33.40
// ms; PAPER mode is 1% faster without).
template <bool UNITE>
__device__ __noinline__ void overflow_row_cc(Smem &S, const Params &p, uint32_t pb, int o, int dy, int nb) {
    overflow_row_in<TPX_MODE_CC, UNITE>(S, p, pb, o, dy, nb);
}
template <int MODE, bool UNITE>
__device__ __forceinline__ void overflow_row(Smem &S, const Params &p, uint32_t pb, int o, int dy, int nb) {
    if constexpr (MODE == TPX_MODE_CC) overflow_row_cc<UNITE>(S, p, pb, o, dy, nb);
    else overflow_row_in<MODE, UNITE>(S, p, pb, o, dy, nb);
}

// One warp resolves the record offset of tile tl holding nc records
// (decoupled look-back over the counts), publishes its inclusive count and,
// for the last tile, the call's totals; the offsets come back in *O. In a
// batch the chain also carries the tile's nt triggers, and a run's first tile
// records the run's record and trigger offsets.
// Without `block`, gives up (false, nothing published) when a predecessor's
// count is not out yet.
template <bool BATCH>
__device__ bool resolve_offset(const Params &p, unsigned seq, long long tl, int nc, long long ntr, int nt, int run,
                               bool run_first, bool block, longlong2 *O) {
    unsigned st2 = 0;
    longlong2 Ow = make_longlong2(0, 0);
    bool ready = true;
    if (tl > 0) Ow = lookback_count_warp<BATCH>(p, tl, seq, &st2, block, &ready);
    if (!ready) return false;
    if ((threadIdx.x & 31) == 0) {
        if (tl > 0 && tl + 1 != p.hold) {
            __stcg(&p.ts.cpre[tl], Ow.x + (long long)nc);
            if (BATCH) __stcg(&p.bt.tcpre[tl], Ow.y + (long long)nt);
            st_release(&p.ts.cflags[tl], (seq << 2) | 2u);
        }
        if (BATCH && run_first) {
            p.bt.run_rec_off[run] = Ow.x;
            p.bt.run_trig_off[run] = Ow.y;
        }
        if (tl == p.n_tiles - 1) {
            const long long nt_all = BATCH ? Ow.y + nt : ntr;
            *p.n_clusters = Ow.x + nc;
            *p.n_trig = nt_all;
            if (BATCH) {
                p.bt.run_rec_off[p.bt.n_runs] = Ow.x + nc;
                p.bt.run_trig_off[p.bt.n_runs] = nt_all;
            }
            if (Ow.x + nc > p.cl_cap) atomicOr(&p.ctl->status, ST_CLUSTER_CAP);
            if (nt_all > p.trig_cap) atomicOr(&p.ctl->status, ST_TRIG_CAP);
        }
    }
    *O = Ow;
    return true;
}

// Copies a finished tile's staged records (in label order) and, in a batch,
// its trigger times to their offset, by the service warp: coalesced, eight
// loads in flight per lane. False: a predecessor's count is not out yet (and
// `block` not set); the caller tries again.
template <bool BATCH>
__device__ bool copy_out(Smem &S, const Params &p, unsigned seq, int slot, bool block) {
    constexpr int NP = BATCH ? RING : 1;
    const int lane = threadIdx.x & 31;
    constexpr int WPR = (int)(sizeof(tpx_record) / 8);
    const long long pt = S.pend[slot].tile, ntr = S.pend[slot].ntr;
    const int nc = S.pend[slot].ncl, nt = S.pend[slot].ntdc, run = S.pend[slot].run;
    const bool first = S.pend[slot].first, big = S.pend[slot].big;
    longlong2 Ow;
    if (!resolve_offset<BATCH>(p, seq, pt, nc, ntr, nt, run, first, block, &Ow)) return false;
    const long long O = Ow.x;
    const long long keep = min((long long)nc, max(0LL, p.cl_cap - O));
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(
        (BATCH && big) ? br_stage(p, slot)
                       : p.stage + (STAGED_ONLY ? S.pend[slot].at : ((long long)blockIdx.x * NP + slot) * C));
    if (p.rec64) {   // 64-byte records: the first 8 words of each staged record
        unsigned long long *d64 = reinterpret_cast<unsigned long long *>(p.clusters) + O * 8;
        const long long nw = keep * 8;
        for (long long w0 = lane; w0 < nw; w0 += 32 * 8) {
            unsigned long long v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const long long w = w0 + 32 * u;
                v[u] = w < nw ? __ldcg(src + (w >> 3) * WPR + (w & 7)) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (w0 + 32 * u < nw) d64[w0 + 32 * u] = v[u];
        }
    }
    unsigned long long *dst = reinterpret_cast<unsigned long long *>(p.clusters + O);
    const long long nw = p.rec64 ? 0 : keep * WPR;
    for (long long w0 = lane; w0 < nw; w0 += 32 * 8) {
        unsigned long long v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = w0 + 32 * u < nw ? __ldcg(src + w0 + 32 * u) : 0ull;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (w0 + 32 * u < nw) dst[w0 + 32 * u] = v[u];
    }
    if (BATCH) {
        const long long TO = Ow.y;
        const long long tkeep = min((long long)nt, max(0LL, p.trig_cap - TO));
        const long long *ts = p.bt.tstage + ((long long)blockIdx.x * NP + slot) * T;
        for (long long i = lane; i < tkeep; i += 32) p.trig[TO + i] = __ldcg(ts + i);
    }
    __syncwarp();
    return true;
}

// the exact integer moments of one cluster from its member list (Sec. V.C)
// and its canonical label: the earliest member in (time, position) order
struct Moments {
    long long s_tt;                    // sum of ToT x biased ToF
    uint32_t s_tot, s_x, s_y;          // a range's sums fit 32 bits (C x 1023 x 255 < 2^32)
    int n, npk;
    int seg;                           // its shot, as a trigger index of the range
    uint32_t best_lo;                  // label position
    int tofb0;                         // its biased ToF
};
static_assert((unsigned long long)C * 1023 * 255 < (1ull << 32), "32-bit moment sums");

__device__ __forceinline__ Moments walk_members(const Smem &S, const Params &p, uint32_t head) {
    uint64_t best = ~0ull;
    Moments m{0, 0, 0, 0, 0, 0, 0, 0, 0};
    // the next member's words are on their way while this one is added up
    uint32_t k = head;
    if (!TPX_IN(k, C)) return m;
    uint64_t rm = S.srec[k];
    uint32_t pos = S.spos[k], dimmed = S.notpeak[k];
    m.seg = r_seg(rm);
    for (;;) {
        const uint32_t nx = S.u2.mnext[k];
        const bool more = nx != EMPTY && TPX_IN(nx, C);
        const uint32_t kn = more ? nx : k;
        const uint64_t rn = S.srec[kn];
        const uint32_t pn = S.spos[kn], dn = S.notpeak[kn];
        const uint32_t tot = (uint32_t)r_tot(rm), tf = (uint32_t)r_tof(rm);
        best = min(best, ((uint64_t)tf << 16) | pos);
        m.n += 1;
        m.npk += dimmed ? 0 : 1;
        m.s_tot += tot;
        m.s_x += tot * (uint32_t)r_x(rm);
        m.s_y += tot * (uint32_t)r_y(rm);
        m.s_tt += (long long)((uint64_t)tot * tf);
        if (!more) break;
        k = nx;
        rm = rn;
        pos = pn;
        dimmed = dn;
    }
    m.best_lo = (uint32_t)(best & 0xFFFFu);
    m.tofb0 = (int)(best >> 16);
    return m;
}

// the record of a cluster whose label pixel lies at position best_lo of the
// range at stream position base
__device__ __forceinline__ tpx_record make_record(const Moments &m, const Smem &S, const Params &p, long long base,
                                                  long long shot0) {
    const long long tofc0 = (long long)m.tofb0 - kTofBias;
    const long long s_t = m.s_tt - (long long)m.tofb0 * (long long)m.s_tot;
    tpx_record o;
    o.label = p.idx_base + base + m.best_lo;
    o.shot = shot0 + m.seg;
    o.t0 = S.tdc_t[m.seg] + tofc0;
    o.s_tot = m.s_tot; o.s_x = m.s_x; o.s_y = m.s_y; o.s_t = s_t;
    o.n = m.n; o.n_peaks = m.npk;
    com_from_moments(o.s_x, o.s_y, s_t, o.s_tot, tofc0, &o.x, &o.y, &o.tof);
    return o;
}

// a record at position idx of the caller's buffer (88 bytes, or its first 64
// with TPX_FLAG_RECORDS64)
__device__ __forceinline__ void out_record(const Params &p, long long idx, const tpx_record &o) {
    if (p.rec64) {
        const unsigned long long *w = reinterpret_cast<const unsigned long long *>(&o);
        unsigned long long *d = reinterpret_cast<unsigned long long *>(p.clusters) + idx * 8;
#pragma unroll
        for (int k = 0; k < 8; ++k) d[k] = w[k];
    } else {
        p.clusters[idx] = o;
    }
}

// rank of label position lp among the tile's labels (after the bitmap scan)
__device__ __forceinline__ int label_rank(const Smem &S, uint32_t lp) {
    return (int)S.u4.lpre[lp >> 5] + __popc(S.u3.lbits[lp >> 5] & ((1u << (lp & 31)) - 1u));
}

// the labels before each bitmap word, by one warp
__device__ __forceinline__ void scan_label_bits(Smem &S) {
    constexpr int WPL = C / 32 / 32;   // bitmap words per lane
    const int lane = threadIdx.x & 31;
    int c = 0;
#pragma unroll
    for (int k = 0; k < WPL; ++k) c += __popc(S.u3.lbits[lane * WPL + k]);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    int run = incl - c;
#pragma unroll
    for (int k = 0; k < WPL; ++k) {
        S.u4.lpre[lane * WPL + k] = (uint16_t)run;
        run += __popc(S.u3.lbits[lane * WPL + k]);
    }
}

// ------------------------------------------------------------- big ranges
// A range longer than the range capacity C (in CC mode: a shot of more pixels
// than a tile holds) stays in the launch. The CTA decodes the whole range
// into its own global scratch (the tile's unwrap, binning and cut, Sec.
// IV.A-C), sorts the kept pixels by (shot, time bin, 8-column x stripe), so
// that a cluster's pixels lie together, and chains them by cell in a hash. Each
// pixel walks the chains of the forward half of its box (in its own cell only
// the pixels before it in the sorted order), so every adjacent pair (Sec. V.A:
// same shot, box neighbours, |dt| within the radius) is seen once. (Comparing
// each pixel with all of the time bins and stripes around it, as wide boxes
// still do, cost 134 of 179 warp instructions per packet.) Union-find over the sorted order
// runs in shared
// memory (16-bit parents, roots linked by a hashed priority). The
// exact integer moments of each cluster (Sec. V.C) are gathered with
// warp-aggregated atomics, and the records are staged in label order in the
// scratch (copied out like a tile's). A range this cannot hold either goes
// back to the general path with its run: more than BR_L positions, BR_N
// kept pixels or BR_S shots.
// 16-bit parents addressed in the shared window (pb: the array's shared
// address), as the tile's union-find addresses its words
__device__ __forceinline__ unsigned br_ld(uint32_t pb, unsigned x) {
    unsigned short v;
    asm volatile("ld.volatile.shared.u16 %0, [%1];" : "=h"(v) : "r"(pb + 2 * x) : "memory");
    return v;
}
__device__ __forceinline__ void br_st(uint32_t pb, unsigned x, unsigned v) {
    asm volatile("st.volatile.shared.u16 [%0], %1;" ::"r"(pb + 2 * x), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ unsigned br_cas(uint32_t pb, unsigned x, unsigned cmp, unsigned v) {
    unsigned short o;
    asm volatile("atom.shared.cas.b16 %0, [%1], %2, %3;"
                 : "=h"(o) : "r"(pb + 2 * x), "h"((unsigned short)cmp), "h"((unsigned short)v) : "memory");
    return o;
}
__device__ __forceinline__ void br_or(uint32_t a, unsigned v) {
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned br_find(uint32_t pb, unsigned x) {
    for (;;) {
        const unsigned px = br_ld(pb, x);
        if (px == x) return x;
        const unsigned g = br_ld(pb, px);
        if (g == px) return px;
        br_st(pb, x, g);   // path halving: g is an ancestor of x
        x = g;
    }
}
__device__ __forceinline__ unsigned br_root(uint32_t pb, unsigned x) {   // changes nothing
    unsigned px;
    while ((px = br_ld(pb, x)) != x) x = px;
    return x;
}
// The root of a big-range cluster need not be any particular pixel (its
// label comes from its moments), so roots are linked by a hashed priority,
// the lower under the higher: the sorted order puts a cluster's pixels on
// consecutive slots, and linking by slot would chain them. Links always rise
// in (priority, slot) order, so the forest stays acyclic.
__device__ __forceinline__ unsigned br_prio(unsigned x) { return ((x * 0x9E3779B1u) & 0xFFFF0000u) | x; }
__device__ __forceinline__ void br_unite(uint32_t pb, unsigned a, unsigned b) {
    for (;;) {
        a = br_find(pb, a);
        b = br_find(pb, b);
        if (a == b) return;
        const bool a_low = br_prio(a) < br_prio(b);
        const unsigned child = a_low ? a : b, up = a_low ? b : a;
        const unsigned old = br_cas(pb, child, child, up);
        if (old == child) return;
        if (a_low) a = old; else b = old;   // the child was linked meanwhile
    }
}

// The range that starts at stream position `base` (first trigger packet at f,
// the next one not before `from`): its cluster count, or -1 with a status bit set when it goes back to
// the general path. Called by every thread of the CTA after the tile's
// staging slot is free; writes the labels, local-maximum flags and staged
// records, and replaces the tile's keep / drop counts by the whole range's.
#ifdef TPX_PHASE_TIMING
#define BR_PH(k)                                                                          \
    do {                                                                                  \
        const long long ph_now = clock64();                                               \
        if ((threadIdx.x & 31) == 0) atomicAdd(&S.ph[k], (unsigned long long)(ph_now - br_t)); \
        br_t = ph_now;                                                                    \
    } while (0)
#else
#define BR_PH(k) do {} while (0)
#endif
// What the window pass needs of a big range: its sorted pixels, the ends of
// their keys (bins), the shots' first bins, times and bin widths.
struct BrSorted {
    const uint64_t *srec;
    const uint16_t *spos;
    const unsigned *bins;
    const int *lo, *b0, *w;
    uint64_t *sbuf;
    int *task;
    uint32_t pb, nb_sh;
    int N, NS, SW;
};
// The earlier pixels that can neighbour pixel i: two runs of consecutive slots,
// the previous time bin's stripes around its own, and its own bin's left stripe
// with its own key up to itself.
__device__ __forceinline__ void br_candidates(const BrSorted &V, int i, uint64_t r, int *a0, int *la, int *b0, int *lb) {
    const int s = r_seg(r), st = r_x(r) / V.SW;
    const int bin = V.b0[s] + (r_tof(r) - V.lo[s]) / V.w[s];
    auto first = [&](int k) -> int { return k > 0 ? (int)V.bins[k - 1] : 0; };   // a key's first slot
    *a0 = *la = 0;
    if (bin > V.b0[s]) {
        *a0 = first((bin - 1) * V.NS + max(st - 1, 0));
        *la = (int)V.bins[(bin - 1) * V.NS + min(st + 1, V.NS - 1)] - *a0;
    }
    *b0 = first(bin * V.NS + max(st - 1, 0));
    *lb = i - *b0;
}
// The neighbour pass of wide boxes: every pixel is compared with the pixels of
// its window, whatever the radii; an adjacent pair clears the loser's
// local-maximum flag and unites. A warp takes 32 consecutive pixels at a time,
// the next task from the chunk's counter, and spreads all their (pixel,
// candidate) pairs evenly over its lanes: a prefix of the pixels' counts, and
// each lane finds the pixel of its pair by a search over the lanes.
__device__ __noinline__ void br_window(const Params &p, const BrSorted V) {
    const int tid = threadIdx.x, lane = tid & 31, rx = p.rx, ry = p.ry, dt = p.dt;
    for (int a = 0; a < V.N; a += BR_CH) {
        const int e = min(V.N, a + BR_CH);
        int lo;   // the chunk's pixels look no further back than the start of the first one's previous bin
        {
            const uint64_t ra = V.srec[a];
            const int s = r_seg(ra), bin = V.b0[s] + (r_tof(ra) - V.lo[s]) / V.w[s];
            const int k0 = (bin > V.b0[s] ? bin - 1 : bin) * V.NS;
            lo = k0 > 0 ? (int)V.bins[k0 - 1] : 0;
        }
        const bool fits = e - lo <= BR_SB;
        if (tid == 0) *V.task = 0;
        if (fits)
            for (int j = lo + tid; j < e; j += NTW) V.sbuf[j - lo] = V.srec[j];
        cta_sync();
        auto rec_at = [&](int j) -> uint64_t { return fits ? V.sbuf[j - lo] : V.srec[j]; };
        const int ntask = (e - a + 31) >> 5;
        for (;;) {
            int task = 0;
            if (lane == 0) task = atomicAdd(V.task, 1);
            task = __shfl_sync(0xffffffffu, task, 0);
            if (task >= ntask) break;
            const int i0 = a + 32 * task, i = i0 + lane;
            int a0 = 0, na = 0, c0 = 0, nc = 0;
            if (i < e) br_candidates(V, i, rec_at(i), &a0, &na, &c0, &nc);
            const int n = na + nc;
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            const int off = incl - n;
            const int W = __shfl_sync(0xffffffffu, incl, 31);
            for (int wb = 0; wb < W; wb += 32) {
                const int w = wb + lane;
                int q = 0;   // the last lane whose pairs start at or before w
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int o = __shfl_sync(0xffffffffu, off, q + step);
                    if (o <= w) q += step;
                }
                const int qa0 = __shfl_sync(0xffffffffu, a0, q), qna = __shfl_sync(0xffffffffu, na, q);
                const int qc0 = __shfl_sync(0xffffffffu, c0, q), qoff = __shfl_sync(0xffffffffu, off, q);
                if (w >= W) continue;
                const int c = w - qoff, ip = i0 + q, j = c < qna ? qa0 + c : qc0 + (c - qna);
                if (!TPX_IN(j, V.N) || !TPX_IN(ip, V.N)) continue;
                const uint64_t rp = rec_at(ip), rj = rec_at(j);
                const int dx = r_x(rj) - r_x(rp), dy = r_y(rj) - r_y(rp);
                if (dx < -rx || dx > rx || dy < -ry || dy > ry || !within(r_tof(rj) - r_tof(rp), dt)) continue;
                const int tj = r_tot(rj), ti = r_tot(rp);
                const bool j_wins = tj > ti || (tj == ti && V.spos[j] > V.spos[ip]);
                const int loser = j_wins ? ip : j;
                br_or(V.nb_sh + 4 * (loser >> 5), 1u << (loser & 31));
                br_unite(V.pb, (unsigned)ip, (unsigned)j);
            }
        }
        cta_sync();
    }
}

template <bool BATCH>
__device__ __noinline__ int big_range(Smem &S, const Params &p, long long base, long long rend, int f, int from,
                                      bool prev_global, const GAgg &E, int slot) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
#ifdef TPX_PHASE_TIMING
    long long br_t = clock64();
#endif
    const long long tp = p.thr_pix, tt = p.thr_tdc;
    unsigned char *R = reinterpret_cast<unsigned char *>(&S);
    uint16_t *par = reinterpret_cast<uint16_t *>(R);
    unsigned *npk = reinterpret_cast<unsigned *>(R + 2 * BR_N);
    unsigned *bins = npk + BR_N / 32;
    unsigned *lbits = bins + BR_BINS + 4;
    uint16_t *lpre = reinterpret_cast<uint16_t *>(lbits + BR_LW);
    int *sg_n = reinterpret_cast<int *>(lpre + BR_LW);
    int *sg_lo = sg_n + BR_S, *sg_hi = sg_lo + BR_S, *sg_b0 = sg_hi + BR_S, *sg_w = sg_b0 + BR_S;
    // misc: [0..2] range-end slots, [3] first pixel, [4] kept, [5] dropped
    // before a trigger, [6] background, [7] failure bits, [8] clusters, [9] peaks
    int *misc = sg_w + BR_S;
    uint16_t *nx_sh = reinterpret_cast<uint16_t *>(misc + 16);   // [BR_NX] the cell chains
    unsigned char *G = p.big + (size_t)blockIdx.x * BR_STRIDE;
    uint64_t *g_rec = reinterpret_cast<uint64_t *>(G);
    uint64_t *g_srec = g_rec + (BR_L + 1);
    uint16_t *g_spos = reinterpret_cast<uint16_t *>(g_srec + BR_N);
    BrMom *g_mom = reinterpret_cast<BrMom *>(g_spos + BR_N);
    // before the moments: up to three further neighbours per pixel, and the
    // cell chains past BR_NX
    uint64_t *g_more = reinterpret_cast<uint64_t *>(g_mom);
    uint16_t *nx_g = reinterpret_cast<uint16_t *>(g_more + BR_N);
    const uint32_t pb = (uint32_t)__cvta_generic_to_shared(par);      // shared addresses
    const uint32_t nb_sh = (uint32_t)__cvta_generic_to_shared(npk);
    const int rx = p.rx, ry = p.ry, dtr = p.dt;
    cta_sync();
    if (tid < 16) misc[tid] = tid < 4 ? INT_MAX : 0;
    cta_sync();

    // ---- the range end: the first TDC packet at or past `from` (the pre-pass
    // found none in between); four packets per thread per step, the
    // steps' minima rotating over three slots as in the tile's look-ahead ----
    int L = 0;
    bool term = false;
    {
        constexpr int STEP = 4 * NTW;
        long long q0 = from;
        for (int k = 0;; ++k) {
            const long long lim = min((long long)BR_L, rend - base);
            if (q0 >= lim) { L = (int)lim; break; }
            if (tid == 0) misc[(k + 1) % 3] = INT_MAX;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const long long q = q0 + u * NTW + tid;
                if (q < lim && (__ldcg(p.pk + base + q) >> 60) == 0x6u) atomicMin(&misc[k % 3], (int)q);
            }
            cta_sync();
            const int lf = misc[k % 3];
            if (lf != INT_MAX) { L = lf + 1; term = true; break; }
            q0 += STEP;
        }
    }
    // not terminated before the position limit while the run goes on
    if (!term && base + L < rend) { if (tid == 0) atomicOr(&S.status, ST_CAPACITY); return -1; }

    // ---- walk 2 over [0, L): wrap steps and TDC counts per contiguous chunk ----
    const int kpd = (L + NTW - 1) / NTW;
    const int p0 = tid * kpd;
    int ntd = 0, jp = 0;
    {
        int lpx = -1, fpx = INT_MAX;
        long long lr = 0;
        for (int j0 = 0; j0 < kpd; j0 += 8) {   // eight loads in flight
            uint64_t w8[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w8[u] = j0 + u < kpd && p0 + j0 + u < L ? __ldg(p.pk + base + p0 + j0 + u) : 0ull;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const unsigned h = (unsigned)(w8[u] >> 60);
                if (h == 0xBu) {
                    const long long r = pix_raw(w8[u]);
                    if (lpx >= 0) jp += (int)jump(r - lr, tp); else fpx = p0 + j0 + u;
                    lpx = p0 + j0 + u;
                    lr = r;
                } else if (h == 0x6u) {
                    ++ntd;
                }
            }
        }
        if (lpx >= 0) {
            for (int q = p0 + kpd; q < L; ++q) {
                const uint64_t w = __ldg(p.pk + base + q);
                if ((w >> 60) == 0xBu) { jp += (int)jump(pix_raw(w) - lr, tp); break; }
            }
        }
        const int fw = (int)__reduce_min_sync(0xffffffffu, (unsigned)fpx);
        if (lane == 0 && fw != INT_MAX) atomicMin(&misc[3], fw);
    }
    unsigned pk_tot;
    const unsigned pk_ex = block_scan_vadd2(S, ((unsigned)ntd << 16) | ((unsigned)jp & 0xFFFFu), &pk_tot);
    const int li0 = (int)(pk_ex >> 16);
    const int nseg = (int)(pk_tot >> 16);
    const int jp_ex = (int)(short)(pk_ex & 0xFFFFu);
    if (nseg > BR_S || nseg > MAXSEG) { if (tid == 0) atomicOr(&S.status, ST_CAPACITY); return -1; }
    if (tid == 0) {
        const int fp = misc[3];
        S.j0 = (fp != INT_MAX && E.pix.n > 0) ? jump(pix_raw(__ldcg(p.pk + base + fp)) - E.pix.last, tp) : 0;
    }
    if (ntd) {
        int li = li0;
        for (int j = 0; j < kpd; ++j) {
            const int q = p0 + j;
            if (q >= L) break;
            if ((__ldg(p.pk + base + q) >> 60) != 0x6u) continue;
            S.tdc_pos[li] = (uint16_t)q;
            ++li;
        }
    }
    for (int s = tid; s < nseg; s += NTW) { sg_n[s] = 0; sg_lo[s] = INT_MAX; sg_hi[s] = INT_MIN; }
    cta_sync();
    // the trigger times (one warp, a scan of the TDC wrap steps)
    if (tid < 32) {
        bool has = E.tdc.n > 0;
        long long last = E.tdc.last, ep = E.tdc.sum, t_last = 0;
        for (int i0 = 0; i0 < nseg; i0 += 32) {
            const int i = i0 + lane;
            long long r = 0;
            if (i < nseg) r = tdc_raw(__ldcg(p.pk + base + S.tdc_pos[i]));
            const long long rp = __shfl_up_sync(0xffffffffu, r, 1);
            int st = 0;
            if (i < nseg && (lane > 0 || has)) st = (int)jump(r - (lane > 0 ? rp : last), tt);
            int inc = st;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            const long long t = r + (ep + inc) * kTdcPeriod;
            const long long tp_ = __shfl_up_sync(0xffffffffu, t, 1);
            if (i < nseg) {
                S.tdc_t[i] = t;
                if ((lane > 0 || i0 > 0) && t < (lane > 0 ? tp_ : t_last)) atomicOr(&p.ctl->status, ST_TRIG_ORDER);
            }
            const int lastl = min(31, nseg - 1 - i0);
            ep += __shfl_sync(0xffffffffu, inc, lastl);
            last = __shfl_sync(0xffffffffu, r, lastl);
            t_last = __shfl_sync(0xffffffffu, t, lastl);
            has = true;
        }
    }
    cta_sync();

    BR_PH(20);
    // ---- walk 4 over [0, L): shot, cut, timewalk, packed record per position
    // (the tile's rule), and each shot's kept count and ToF span ----
    {
        long long ep = E.pix.sum + S.j0 + jp_ex;
        bool has = false;
        long long last = 0;
        int seg = li0 - 1;
        const long long t_prev_global = E.tdc.last + E.tdc.sum * kTdcPeriod;
        int c_keep = 0, c_pre = 0, c_bg = 0;
        bool exc = false;
        int cs = -1, cn = 0, clo = INT_MAX, chi = INT_MIN;   // the current shot's running stats
        uint64_t w4[4];
        for (int j = 0; j < kpd; ++j) {
            const int q = p0 + j;
            if (q >= L) break;
            if ((j & 3) == 0) {   // four loads in flight
#pragma unroll
                for (int u = 0; u < 4; ++u) w4[u] = q + u < L ? __ldg(p.pk + base + q + u) : 0ull;
            }
            const uint64_t w = w4[0];
            w4[0] = w4[1]; w4[1] = w4[2]; w4[2] = w4[3];
            const unsigned h = (unsigned)(w >> 60);
            uint64_t rec = INVALID;
            if (h == 0x6u) {
                ++seg;
            } else if (h == 0xBu) {
                const long long r = pix_raw(w);
                if (has) ep += jump(r - last, tp);
                has = true;
                last = r;
                const long long t = r + ep * kPixPeriod;
                if (seg < 0) {
                    if (!prev_global) ++c_pre;
                } else if (seg < nseg) {
                    const long long t_lo = S.tdc_t[seg];
                    const bool has_hi = seg + 1 < nseg;
                    int verdict;                      // 0 keep, 1 bg, 2 pre, 3 undecidable here
                    if (has_hi && t >= S.tdc_t[seg + 1]) verdict = 3;
                    else if (t >= t_lo) verdict = (t - t_lo > p.tof_max) ? 1 : 0;
                    else {
                        const bool hp = seg > 0 || prev_global;
                        const long long tprev = seg > 0 ? S.tdc_t[seg - 1] : t_prev_global;
                        if (!hp) verdict = 2;
                        else if (t >= tprev) verdict = (t - tprev > p.tof_max) ? 1 : 3;
                        else verdict = 3;
                    }
                    if (verdict == 0) {
                        const int tot = pix_tot(w);
                        const long long tc = t - (p.lut ? (long long)p.lut[tot] : 0LL);
                        const int tofb = (int)(tc - t_lo + kTofBias);
                        rec = mkrec((uint32_t)tofb, (uint32_t)seg, (uint32_t)tot, (uint32_t)pix_x(w), (uint32_t)pix_y(w));
                        ++c_keep;
                        if (seg != cs) {
                            if (cs >= 0) { atomicAdd(&sg_n[cs], cn); atomicMin(&sg_lo[cs], clo); atomicMax(&sg_hi[cs], chi); }
                            cs = seg; cn = 0; clo = INT_MAX; chi = INT_MIN;
                        }
                        ++cn;
                        clo = min(clo, tofb);
                        chi = max(chi, tofb);
                    } else if (verdict == 1) ++c_bg;
                    else if (verdict == 2) ++c_pre;
                    else exc = true;
                }
            }
            g_rec[q] = rec;
        }
        if (cs >= 0) { atomicAdd(&sg_n[cs], cn); atomicMin(&sg_lo[cs], clo); atomicMax(&sg_hi[cs], chi); }
        c_keep = (int)warp_sum((unsigned long long)c_keep);
        c_pre = (int)warp_sum((unsigned long long)c_pre);
        c_bg = (int)warp_sum((unsigned long long)c_bg);
        if (lane == 0) {
            atomicAdd(&misc[4], c_keep);
            atomicAdd(&misc[5], c_pre);
            atomicAdd(&misc[6], c_bg);
        }
        if (exc) atomicOr(&misc[7], (int)ST_EXCEPTION);
    }
    cta_sync();
    const int N = misc[4];
    if (misc[7] || N > BR_N) {
        if (tid == 0) atomicOr(&S.status, misc[7] ? (unsigned)misc[7] : ST_CAPACITY);
        return -1;
    }

    BR_PH(21);
    // ---- time bins: each shot gets a share of the bins by its kept count,
    // each bin at least dt + 1 ticks wide (one warp); a key is a (bin,
    // stripe) pair ----
    // stripes at least rx wide; fewer when the shots need the time bins
    // (every shot takes at least one)
    int NS = rx <= 256 / BR_NS ? BR_NS : (rx <= 2 * 256 / BR_NS ? BR_NS / 2 : 1);
    while (NS > 1 && BR_BINS / NS < 2 * nseg) NS = NS > BR_NS / 2 ? BR_NS / 2 : 1;
    const int SW = 256 / NS;   // stripe width (columns)
    const int TB = BR_BINS / NS;   // time bins over all shots
    if (wid == 0) {
        constexpr int SPL = BR_S / 32;   // shots per lane
        int nb[SPL], tot = 0;
#pragma unroll
        for (int k = 0; k < SPL; ++k) {
            const int s = lane * SPL + k;
            const int n = s < nseg ? sg_n[s] : 0;
            nb[k] = s < nseg ? (n > 0 ? 1 + (int)(((long long)(TB - nseg) * n) / N) : 1) : 0;
            tot += nb[k];
        }
        int incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        int b0 = incl - tot;
#pragma unroll
        for (int k = 0; k < SPL; ++k) {
            const int s = lane * SPL + k;
            if (s < nseg) {
                sg_b0[s] = b0;
                const long long span = sg_n[s] > 0 ? (long long)sg_hi[s] - sg_lo[s] + 1 : 1;
                sg_w[s] = (int)max((long long)dtr + 1, (span + nb[k] - 1) / nb[k]);
                if (sg_n[s] == 0) sg_lo[s] = 0;
            }
            b0 += nb[k];
        }
    }
    for (int b = tid; b < BR_BINS; b += NTW) bins[b] = 0u;
    cta_sync();
    auto bin_of = [&](uint64_t r) -> int {
        const int s = r_seg(r);
        return (sg_b0[s] + (r_tof(r) - sg_lo[s]) / sg_w[s]) * NS + r_x(r) / SW;
    };
    // ---- counting sort of the kept pixels by bin ----
    for (int q0 = tid; q0 < L; q0 += 4 * NTW) {   // (here and below: four positions' loads in flight)
        uint64_t r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = q0 + u * NTW < L ? g_rec[q0 + u * NTW] : INVALID;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (r[u] != INVALID) atomicAdd(&bins[bin_of(r[u])], 1u);
    }
    cta_sync();
    {
        constexpr int BPT = (BR_BINS + NTW - 1) / NTW;   // bins per thread, contiguous
        unsigned c[BPT], s = 0;
#pragma unroll
        for (int k = 0; k < BPT; ++k) { c[k] = tid * BPT + k < BR_BINS ? bins[tid * BPT + k] : 0u; s += c[k]; }
        int total;
        unsigned run = (unsigned)block_scan_int(S, (int)s, &total);
#pragma unroll
        for (int k = 0; k < BPT; ++k) { if (tid * BPT + k < BR_BINS) bins[tid * BPT + k] = run; run += c[k]; }
    }
    cta_sync();
    for (int q0 = tid; q0 < L; q0 += 4 * NTW) {
        uint64_t r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = q0 + u * NTW < L ? g_rec[q0 + u * NTW] : INVALID;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (r[u] == INVALID) continue;
            const unsigned slot = atomicAdd(&bins[bin_of(r[u])], 1u);
            if (!TPX_IN(slot, N)) continue;
            g_srec[slot] = r[u];
            g_spos[slot] = (uint16_t)(q0 + u * NTW);
        }
    }
    for (int i = tid; i < N; i += NTW) par[i] = (uint16_t)i;
    for (int w = tid; w < BR_N / 32; w += NTW) npk[w] = 0u;
    cta_sync();
    // Boxes of more than the eight neighbours: the cells of the forward half (13
    // at radius 2, 113 at 7) or the candidates of a window, whichever is less
    // work (a cell costs about as much as eight candidates). 66 shots of 9000
    // pixels: chains 836, 1318, 5187 us at radius 2, 3, 7, windows 495, 526, 545;
    // with a time radius over the whole shot chains 945 at radius 2, windows 2780.
    const int cells = (rx + 1) * (2 * ry + 1) - ry;
    bool window = false;
    if (cells > 5) {
        const BrSorted V{g_srec, g_spos, bins, sg_lo, sg_b0, sg_w, reinterpret_cast<uint64_t *>(nx_sh), &misc[12], pb, nb_sh, N, NS, SW};
        unsigned cand = 0;   // N^2 in all at most
        for (int i = tid; i < N; i += NTW) {
            int a0, la, b0, lb;
            br_candidates(V, i, g_srec[i], &a0, &la, &b0, &lb);
            cand += (unsigned)(la + lb);
        }
        cand = __reduce_add_sync(0xffffffffu, cand);
        if (lane == 0) atomicAdd(reinterpret_cast<unsigned *>(&misc[13]), cand);
        cta_sync();
        window = (unsigned)misc[13] <= 8u * (unsigned)cells * (unsigned)N;
        if (window) br_window(p, V);
    }
    if (!window) {
        // the neighbour pass's flags, a byte each in what the parents leave free:
        // plain stores (as bits, 32 lanes of one cluster met in the same word's
        // atomics: a third of the path's cycles)
        uint8_t *lost = 3 * N + 3 <= 2 * BR_N ? reinterpret_cast<uint8_t *>(par + N) : nullptr;
        if (lost)
            for (int i = tid; i < N; i += NTW) lost[i] = 0;
        // Behind them, and on in the label bitmap's place, a byte hashed from each
        // pixel's cell, as far as that goes (18,592 pixels with 4096-packet tiles):
        // the other cells of a bucket cost no read of their record, which come from
        // L2 (14% hits in L1)
        constexpr int TAG2 = 6 * BR_LW;                              // bytes of lbits and lpre
        const int tag1 = lost ? 2 * (BR_N - N) - N : 0;
        uint8_t *tags1 = reinterpret_cast<uint8_t *>(par + N) + N, *tags2 = reinterpret_cast<uint8_t *>(lbits);
        auto tag_of = [&](uint32_t cell) -> unsigned { return (cell * 0x85EBCA6Bu) >> 24; };
        cta_sync();
        // ---- the cell chains: the last pixel of a bucket first ----
        constexpr unsigned NONE = 0xFFFFu;
        auto bucket = [&](uint32_t cell) -> unsigned { return __umulhi(cell * 0x9E3779B1u, (unsigned)BR_BINS); };
        for (int b = tid; b < BR_BINS; b += NTW) bins[b] = NONE;
        cta_sync();
        for (int i = tid; i < N; i += NTW) {
            const uint32_t cell = r_cell(g_srec[i]);
            const unsigned prev = atomicExch(&bins[bucket(cell)], (unsigned)i);
            if (i < BR_NX) nx_sh[i] = (uint16_t)prev; else nx_g[i] = (uint16_t)prev;
            if (i < tag1) tags1[i] = (uint8_t)tag_of(cell);
            else if (i - tag1 < TAG2) tags2[i - tag1] = (uint8_t)tag_of(cell);
        }
        cta_sync();

        BR_PH(22);
        // ---- neighbour pass: every pixel against the chains of the cells that can
        // hold its neighbours (the box rule, Sec. V.A); an adjacent pair clears the
        // loser's local-maximum flag (Sec. V.B: the larger ToT wins, equal ToT goes
        // to the later pixel). A pixel points to the first neighbour it finds: its
        // own entry only, and pointers go forward in a strict order (cell, then
        // slot), so they form a forest without a single compare-and-swap. The next
        // three neighbours are kept aside. Consecutive slots are mostly one
        // cluster, so a warp's chains are near each other and its records in L1 ----
        // the first pixel from j on along its chain that may be of the cell (own:
        // only those before pixel i), NONE at the end
        auto next_of = [&](int i, uint32_t cell, unsigned j, bool own) -> unsigned {
            const unsigned tag = tag_of(cell);
            while (j != NONE) {
                if (!TPX_IN(j, N)) return NONE;
                const int k = (int)j - tag1;
                const unsigned t = k < 0 ? tags1[j] : k < TAG2 ? tags2[k] : tag;
                if (t == tag && !(own && j >= (unsigned)i)) return j;
                j = j < (unsigned)BR_NX ? nx_sh[j] : nx_g[j];
            }
            return NONE;
        };
        auto link = [&](unsigned j) -> unsigned { return j < (unsigned)BR_NX ? nx_sh[j] : nx_g[j]; };
        // every neighbour of pixel i among the forward half of its box
        auto walk_all = [&](int i, uint64_t ri, auto pair) {
            const int x = r_x(ri), y = r_y(ri), tb = r_tof(ri);
            const uint32_t seg = r_cell(ri) & ~0xFFFFu;
            auto cell_at = [&](int cx, int cy) -> uint32_t { return seg | ((uint32_t)cy << 8) | (uint32_t)cx; };
            auto first_of = [&](int cx, int cy, bool own) -> unsigned {
                if (cx > 255 || cy < 0 || cy > 255) return NONE;
                return next_of(i, cell_at(cx, cy), bins[bucket(cell_at(cx, cy))], own);
            };
            // the chain from its first candidate j on, whose record is r
            auto walk = [&](uint32_t cell, unsigned j, uint64_t r, bool own) {
                while (j != NONE) {
                    if (r_cell(r) == cell && within(r_tof(r) - tb, dtr)) pair(j, r);
                    j = next_of(i, cell, link(j), own);
                    if (j != NONE) r = g_srec[j];
                }
            };
            if (rx == 1 && ry == 1) {   // the five cells' first candidates, then their records together
                unsigned j[5];
                uint64_t r[5];
                j[0] = first_of(x, y, true);
                j[1] = first_of(x, y + 1, false);
                j[2] = first_of(x + 1, y, false);
                j[3] = first_of(x + 1, y - 1, false);
                j[4] = first_of(x + 1, y + 1, false);
#pragma unroll
                for (int k = 0; k < 5; ++k) r[k] = j[k] != NONE ? g_srec[j[k]] : 0ull;
                walk(cell_at(x, y), j[0], r[0], true);
                walk(cell_at(x, y + 1), j[1], r[1], false);
                walk(cell_at(x + 1, y), j[2], r[2], false);
                walk(cell_at(x + 1, y - 1), j[3], r[3], false);
                walk(cell_at(x + 1, y + 1), j[4], r[4], false);
            } else {
                for (int dx = 0; dx <= rx; ++dx)
                    for (int dy = dx == 0 ? 0 : -ry; dy <= ry; ++dy) {
                        const bool own = dx == 0 && dy == 0;
                        const unsigned j = first_of(x + dx, y + dy, own);
                        if (j != NONE) walk(cell_at(x + dx, y + dy), j, g_srec[j], own);
                    }
            }
        };
        for (int i0 = wid * 32; i0 < N; i0 += NTW) {
            const int i = i0 + lane;
            bool own_lost = false;
            if (i < N) {
                const uint64_t ri = g_srec[i];
                const int ti = r_tot(ri);
                unsigned n = 0;
                uint64_t more = 0;
                walk_all(i, ri, [&](unsigned j, uint64_t rj) {
                    const int tj = r_tot(rj);
                    const bool j_wins = tj > ti || (tj == ti && g_spos[j] > g_spos[i]);
                    if (j_wins) own_lost = true;
                    else if (lost) lost[j] = 1;
                    else br_or(nb_sh + 4 * (j >> 5), 1u << (j & 31));
                    if (n == 0) br_st(pb, (unsigned)i, j);
                    else if (n <= 3) more |= (uint64_t)j << (16 * (n - 1));
                    n = min(n + 1, 5u);
                });
                g_more[i] = more | ((uint64_t)n << 48);
            }
            const unsigned w = __ballot_sync(0xffffffffu, own_lost);   // 32 consecutive slots: one word
            if (lane == 0 && w) br_or(nb_sh + 4 * (i0 >> 5), w);
        }
        cta_sync();
        // every pixel to its root, then the pairs that the pointers left out: the
        // two ends have one root already, nearly always (with a union for each of
        // the 4 pairs per pixel, lanes of one cluster met in the same
        // compare-and-swaps and flag words: this pass took 1.1e6 cycles of the
        // path's 1.5e6 per shot of 15,500 pixels, now 0.33e6 of 0.73e6; 600 such
        // shots 4.1 -> 2.35 ms)
        for (int i = tid; i < N; i += NTW) {
            unsigned r = br_ld(pb, (unsigned)i);
            for (unsigned up = br_ld(pb, r); up != r; up = br_ld(pb, r)) r = up;
            br_st(pb, (unsigned)i, r);
        }
        if (lost)
            for (int i0 = wid * 32; i0 < N; i0 += NTW) {
                const unsigned w = __ballot_sync(0xffffffffu, i0 + lane < N && lost[i0 + lane]);
                if (lane == 0 && w) br_or(nb_sh + 4 * (i0 >> 5), w);
            }
        cta_sync();
        for (int i = tid; i < N; i += NTW) {
            const uint64_t more = g_more[i];
            const unsigned n = (unsigned)(more >> 48);
            auto join = [&](unsigned j) {
                if (TPX_IN(j, N) && br_ld(pb, (unsigned)i) != br_ld(pb, j)) br_unite(pb, (unsigned)i, j);
            };
            if (n <= 4) {
                for (unsigned k = 1; k < n; ++k) join((unsigned)(more >> (16 * (k - 1))) & 0xFFFFu);
            } else {
                walk_all(i, g_srec[i], [&](unsigned j, uint64_t) { join(j); });
            }
        }
    }
    cta_sync();
    for (int w = tid; w < BR_LW; w += NTW) lbits[w] = 0u;
    BR_PH(23);
    // compress: every pixel points to its root. Each pointer is changed by its own
    // thread alone: a find that halves paths on the way could put an ancestor back
    // over a root that the pixel's thread has just stored
    for (int i = tid; i < N; i += NTW) br_st(pb, (unsigned)i, br_root(pb, (unsigned)i));
    cta_sync();
    // roots: their moment records cleared, counted
    {
        int k = 0;
        for (int i = tid; i < N; i += NTW) {
            if (par[i] != i) continue;
            ++k;
            unsigned long long *m = reinterpret_cast<unsigned long long *>(&g_mom[i]);
#pragma unroll
            for (int u = 0; u < 5; ++u) __stcg(m + u, u == 4 ? ~0ull : 0ull);
            __stcg(m + 5, 0ull);
        }
        k = (int)warp_sum((unsigned long long)k);
        if (lane == 0 && k) atomicAdd(&misc[8], k);
    }
    cta_sync();
    const int K = misc[8];

    BR_PH(24);
    // ---- moments: a warp's lanes sharing a root add up among themselves, one
    // lane per root adds to its record ----
    for (int i0 = wid * 32; i0 < N; i0 += NTW) {
        const int i = i0 + lane;
        const bool v = i < N;
        const unsigned r = v ? par[i] : 0xFFFFFFFFu;
        const uint64_t ri = v ? g_srec[i] : 0ull;
        const unsigned pos = v ? g_spos[i] : 0u;
        const unsigned tot = (unsigned)r_tot(ri), tofb = (unsigned)r_tof(ri);
        const unsigned ux = tot * (unsigned)r_x(ri), uy = tot * (unsigned)r_y(ri);
        const unsigned long long utt = (unsigned long long)tot * tofb;
        const bool pk = v && !((npk[i >> 5] >> (i & 31)) & 1u);
        unsigned act = __ballot_sync(0xffffffffu, v);
        unsigned c_pk = 0;
        while (act) {
            const int ld = __ffs(act) - 1;
            const unsigned r0 = __shfl_sync(0xffffffffu, r, ld);
            const bool mine = v && r == r0;
            const unsigned grp = __ballot_sync(0xffffffffu, mine);
            const unsigned a_tot = __reduce_add_sync(0xffffffffu, mine ? tot : 0u);
            const unsigned a_x = __reduce_add_sync(0xffffffffu, mine ? ux : 0u);
            const unsigned a_y = __reduce_add_sync(0xffffffffu, mine ? uy : 0u);
            const unsigned a_tl = __reduce_add_sync(0xffffffffu, mine ? (unsigned)(utt & 0xFFFFFFu) : 0u);
            const unsigned a_th = __reduce_add_sync(0xffffffffu, mine ? (unsigned)(utt >> 24) : 0u);
            const unsigned m_t = __reduce_min_sync(0xffffffffu, mine ? tofb : 0xFFFFFFFFu);
            const unsigned m_p = __reduce_min_sync(0xffffffffu, (mine && tofb == m_t) ? pos : 0xFFFFFFFFu);
            const unsigned n_pk = __popc(__ballot_sync(0xffffffffu, mine && pk));
            if (lane == ld && TPX_IN(r0, N)) {
                BrMom &M = g_mom[r0];
                atomicAdd(&M.s_tot, (unsigned long long)a_tot);
                atomicAdd(&M.s_x, (unsigned long long)a_x);
                atomicAdd(&M.s_y, (unsigned long long)a_y);
                atomicAdd(&M.s_tt, ((unsigned long long)a_th << 24) + a_tl);
                atomicMin(&M.best, ((unsigned long long)m_t << 16) | m_p);
                atomicAdd(&M.n, (unsigned)__popc(grp));
                atomicAdd(&M.npk, n_pk);
            }
            c_pk += n_pk;
            act &= ~grp;
        }
        if (lane == 0 && c_pk) atomicAdd(&misc[9], (int)c_pk);
    }
    cta_sync();
    BR_PH(25);
    // ---- the labels (each cluster's earliest pixel in (time, position)
    // order) marked in the bitmap, then their ranks ----
    for (int i = tid; i < N; i += NTW) {
        if (par[i] != i) continue;
        const unsigned lp = (unsigned)(__ldcg(&g_mom[i].best) & 0xFFFFu);
        atomicOr(&lbits[lp >> 5], 1u << (lp & 31));
    }
    cta_sync();
    {
        constexpr int WPT = (BR_LW + NTW - 1) / NTW;
        unsigned c[WPT], s = 0;
#pragma unroll
        for (int k = 0; k < WPT; ++k) { c[k] = tid * WPT + k < BR_LW ? (unsigned)__popc(lbits[tid * WPT + k]) : 0u; s += c[k]; }
        int total;
        unsigned run = (unsigned)block_scan_int(S, (int)s, &total);
#pragma unroll
        for (int k = 0; k < WPT; ++k) { if (tid * WPT + k < BR_LW) lpre[tid * WPT + k] = (uint16_t)run; run += c[k]; }
    }
    cta_sync();
    // ---- records, staged in label order ----
    tpx_record *dst = br_stage(p, slot);
    for (int i = tid; i < N; i += NTW) {
        if (par[i] != i) continue;
        const unsigned long long *m = reinterpret_cast<const unsigned long long *>(&g_mom[i]);
        const long long s_tot = (long long)__ldcg(m), s_x = (long long)__ldcg(m + 1), s_y = (long long)__ldcg(m + 2);
        const long long s_tt = (long long)__ldcg(m + 3);
        const unsigned long long best = __ldcg(m + 4), nn = __ldcg(m + 5);
        const unsigned lp = (unsigned)(best & 0xFFFFu);
        const int tofb0 = (int)(best >> 16);
        const int k = (int)lpre[lp >> 5] + __popc(lbits[lp >> 5] & ((1u << (lp & 31)) - 1u));
        if (!TPX_IN(k, K) || !TPX_IN(lp, L)) continue;
        const int seg = r_seg(g_rec[lp]);
        const long long tofc0 = (long long)tofb0 - kTofBias;
        tpx_record o;
        o.label = p.idx_base + base + lp;
        o.shot = E.tdc.n + seg;
        o.t0 = S.tdc_t[seg] + tofc0;
        o.s_tot = s_tot; o.s_x = s_x; o.s_y = s_y;
        o.s_t = s_tt - (long long)tofb0 * s_tot;
        o.n = (int)(nn & 0xFFFFFFFFu);
        o.n_peaks = (int)(nn >> 32);
        com_from_moments(o.s_x, o.s_y, o.s_t, s_tot, tofc0, &o.x, &o.y, &o.tof);
        dst[k] = o;
    }
    // ---- per-packet outputs over the range's label span ----
    if (p.labels || p.labels32 || p.is_peak) {
        for (int i0 = tid; i0 < N; i0 += 4 * NTW) {
            unsigned q4[4], lp4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * NTW;
                q4[u] = i < N ? g_spos[i] : 0u;
                lp4[u] = i < N ? (unsigned)(__ldcg(&g_mom[par[i]].best) & 0xFFFFu) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * NTW;
                if (i >= N) break;
                const long long q = q4[u];
                const unsigned lp = lp4[u];
                const uint8_t pk = ((npk[i >> 5] >> (i & 31)) & 1u) ? 0 : 1;
                if (!TPX_IN(base + q, rend)) continue;
                if (p.labels) p.labels[base + q] = p.idx_base + base + lp;
                else if (p.labels32) p.labels32[base + q] = (int)(p.idx_base - p.lab32_base + base + lp);
                if (p.is_peak) p.is_peak[base + q] = pk;
            }
        }
        const int W0 = prev_global ? f : 0, W1 = term ? L - 1 : L;
        for (int q0 = W0 + tid; q0 < W1; q0 += 4 * NTW) {
            uint64_t r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) r[u] = q0 + u * NTW < W1 ? g_rec[q0 + u * NTW] : 0ull;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = q0 + u * NTW;
                if (q >= W1 || r[u] != INVALID || !TPX_IN(base + q, rend)) continue;
                if (p.labels) p.labels[base + q] = -1LL;
                else if (p.labels32) p.labels32[base + q] = -1;
                if (p.is_peak) p.is_peak[base + q] = 0;
            }
        }
    }
    cta_sync();
    BR_PH(26);
    if (tid == 0) {
        S.cnt[C_KEPT] = (unsigned long long)misc[4];
        S.cnt[C_DROP_PRE] = (unsigned long long)misc[5];
        S.cnt[C_DROP_BG] = (unsigned long long)misc[6];
        S.cnt[C_PEAKS] += (unsigned long long)misc[9];
    }
    cta_sync();
    return K;
}

// ------------------------------------------------------------------- kernel
// The service warp plans a tile's range and loads the unwrap state before it: the
// tile's first TDC packet, the first one past the tile (the range's end) from
// the pre-pass's tile table -- a range within the capacity reaches no further
// than LOOK tiles after its own -- and whether a pixel wrap is near.
template <bool BATCH>
__device__ void plan_tile(Smem::Plan &P, const Params &p, long long tile, bool bigr) {
    const int lane = threadIdx.x & 31;
    if (lane == 0) P.tile = tile;
    if (tile >= p.n_tiles) return;
    long long tile0 = 0, tile_end = p.n_tiles, base = tile * T, rend = p.n;
    if (BATCH) {
        const int run = p.bt.tile_run[tile];
        tile0 = p.bt.run_tile0[run];
        if (run + 1 < p.bt.n_runs) tile_end = p.bt.run_tile0[run + 1];
        base = p.bt.run_off[run] + (tile - tile0) * T;
        rend = p.bt.run_off[run + 1];
    }
    if (lane < 8)
        reinterpret_cast<long long *>(&P.E)[lane] = __ldcg(reinterpret_cast<const long long *>(&p.ts.pre[tile]) + lane);
    int f = -1;
    unsigned wrap = 0;
    if (lane <= LOOK && tile + lane < tile_end) {
        const int2 v = __ldcg(reinterpret_cast<const int2 *>(p.ts.tinfo) + tile + lane);
        f = v.x;
        wrap = (unsigned)v.y;
    }
    __syncwarp();
    const unsigned has = __ballot_sync(0xffffffffu, f >= 0) & ~1u;
    const int j = has ? __ffs(has) - 1 : LOOK;       // tiles the range reaches into
    const int fj = __shfl_sync(0xffffffffu, f, j), f0 = __shfl_sync(0xffffffffu, f, 0);
    const unsigned slow = __ballot_sync(0xffffffffu, wrap != 0 && lane <= j);
    if (lane == 0) {
        const long long trig_base = (!BATCH && p.E0) ? p.E0->tdc.n : 0;
        const bool prev_global = P.E.tdc.n > trig_base;
        const int cnt = (int)max(0LL, min((long long)T, rend - base));
        const int w0 = prev_global && f0 >= 0 ? f0 : 0;
        long long len = 0;
        bool term = false, over = false;
        if (f0 >= 0) {
            // the capacity counts from the tile's first packet: a tile's
            // range either always fits or never does, whatever precedes it
            if (has) {
                len = (long long)j * T + fj + 1;
                term = true;
            } else {
                over = tile + LOOK + 1 < tile_end;
                len = over ? C : rend - base;
            }
            if (len > C) { over = true; len = C; term = false; }
            len -= w0;
        } else if (!prev_global) {
            len = cnt;   // before the call's first trigger: nothing to cluster, labels of -1
        }
        P.f = f0;
        P.w0 = w0;
        P.len = (int)len;
        P.term = term ? 1 : 0;
        P.slow = slow != 0 ? 1 : 0;
        P.status = over ? (bigr ? ST_BIG : ST_CAPACITY) : 0u;
        // its packets start moving into L2 (one bulk prefetch, 16-byte granules)
        if (p.l2_prefetch && len > 0) {
            const uint64_t *a = p.pk + ((base + w0) & ~1LL);
            const long long m = min(len + 1, p.n - ((base + w0) & ~1LL)) & ~1LL;
            if (m > 0)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)(8 * m)) : "memory");
        }
    }
}

// The service warp: claims and plans the tile after the one in work, and
// copies finished tiles' records out in order while the workers go on. A
// predecessor's count that is not out yet is tried again later, so a tile
// behind a slow one holds up neither the planning nor (while the ring has
// room) the workers. On the large batch the copy of a tile takes about 9k
// cycles, nearly all latency of the look-back and of the copies; as one of the
// workers' phases it was 11% of the kernel.
template <int MODE, bool BATCH>
__device__ void service(Smem &S, const Params &p, unsigned seq, bool bigr) {
    constexpr int NP = BATCH ? RING : 1;
    const int lane = threadIdx.x & 31;
    int planned = 0, consumed = 0, last = -1;
    long long tries = 0, idle = 0;
    for (;;) {
        int produced = 0, entries = 0;
        if (lane == 0) {
            produced = *reinterpret_cast<volatile int *>(&S.produced);
            __threadfence_block();
            entries = *reinterpret_cast<volatile int *>(&S.entries);   // at least those of the tiles seen finished
        }
        produced = __shfl_sync(0xffffffffu, produced, 0);
        entries = __shfl_sync(0xffffffffu, entries, 0);
        bool did = false;
        if (last < 0 && planned < produced + 2) {
            unsigned claim = 0;
            if (lane == 0) claim = atomicAdd(&p.ctl->tile_counter, 1u);
            const long long tile = (long long)__shfl_sync(0xffffffffu, claim, 0);
            plan_tile<BATCH>(S.plan[planned & 1], p, tile, bigr);
            if (tile >= p.n_tiles) last = planned;
            __syncwarp();
            ++planned;
            if (lane == 0) {
                __threadfence_block();
                *reinterpret_cast<volatile int *>(&S.planned) = planned;
            }
            did = true;
        }
        if (consumed < entries) {
            __threadfence_block();
            bool give_up = tries > 0 && timed_out(p);
            if (tries > MAX_TRIES) {
                if (lane == 0) atomicOr(&p.ctl->status, ST_DEVTIMEOUT);
                __threadfence();
                give_up = true;
            }
            give_up = __any_sync(0xffffffffu, give_up);
            if (copy_out<BATCH>(S, p, seq, consumed % NP, give_up)) {
                tries = 0;
                ++consumed;
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    *reinterpret_cast<volatile int *>(&S.consumed) = consumed;
                }
                did = true;
            } else {
                ++tries;
            }
        }
        if (last >= 0 && produced == last && consumed == entries) break;
        if (did) { idle = 0; continue; }
        if (++idle > MAX_HANDOVER) {
            if (lane == 0) atomicOr(&p.ctl->status, ST_DEVTIMEOUT);
            break;
        }
        __nanosleep(BATCH && consumed < entries ? 1000 : 100);
    }
}

// a worker thread waits until a handover count passes `than` (bounded)
__device__ __forceinline__ bool wait_count(const int *count, int than, const Params &p) {
    long long spins = 0;
    while (*reinterpret_cast<const volatile int *>(count) <= than) {
        if (++spins > MAX_HANDOVER) {
            atomicOr(&p.ctl->status, ST_DEVTIMEOUT);
            return false;
        }
        __nanosleep(40);
    }
    __threadfence_block();
    return true;
}

template <int MODE, bool STAGED, bool BATCH>
__global__ void __launch_bounds__(NT, MINB) fused_kernel(const Params p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &S = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const long long tp = p.thr_pix, tt = p.thr_tdc;
    const unsigned seq = p.seq & 0x3FFFFFFFu;
    const uint32_t pb = (uint32_t)__cvta_generic_to_shared(S.par);
    // ranges past the capacity go through the big-range path (CC mode, batches)
    constexpr bool BIGR = BATCH && STAGED && MODE == TPX_MODE_CC;
    constexpr int NP = BATCH ? RING : 1;   // finished tiles a CTA may hold
    if (tid < C_NUM) { S.cnt[tid] = 0; S.acc[tid] = 0; }
    if (tid == 0) S.planned = S.produced = S.entries = S.consumed = 0;
    int ent = 0;   // entries this CTA has made
#ifdef TPX_PHASE_TIMING
    if (tid < 32) S.ph[tid] = 0;
    long long ph_t = clock64();
#endif
    __syncthreads();
    if (wid == NW) {
        service<MODE, BATCH>(S, p, seq, BIGR && p.big);
        return;
    }

    for (int it = 0;; ++it) {
        // the tile's plan; the per-tile fields start over
        const Smem::Plan &P = S.plan[it & 1];
        if (tid == 0) {
            if (!wait_count(&S.planned, it, p)) S.plan[it & 1].tile = p.n_tiles;
            S.status = P.status;
            S.first_pix = INT_MAX;
            S.nroot = S.nov = S.qn = S.rw = 0;
            S.n_pre = S.n_bg = S.n_pk = 0;
        }
        cta_sync();
        const long long tile = P.tile;
        if (tile >= p.n_tiles) {
            // this CTA's counters (packets of each class are counted by the
            // unwrap pre-pass)
            if (tid < C_NUM && tid != C_PIXELS && tid != C_TDCS && tid != C_CORRUPT && S.acc[tid])
                atomicAdd(&p.ctl->counters[tid], S.acc[tid]);
#ifdef TPX_PHASE_TIMING
            TPX_PH(16);
            cta_sync();
            if (tid < 32 && S.ph[tid]) atomicAdd(&g_phase[tid], S.ph[tid]);
#endif
            break;
        }
        // the tile: in a batch, the tile queue names the run (each run is a
        // stream of its own: the chains start over at its first tile)
        int run = 0;
        long long tile0 = 0, rend = p.n, base;
        if (BATCH) {
            run = p.bt.tile_run[tile];
            tile0 = p.bt.run_tile0[run];
            base = p.bt.run_off[run] + (tile - tile0) * T;
            rend = p.bt.run_off[run + 1];
        } else {
            base = tile * T;
        }
        const int cnt = (int)max(0LL, min((long long)T, rend - base));
        // the range: L packets from w0 on, its first TDC packet at R0 (both
        // from w0), the TDC packet that ends it included when there is one
        const int f = P.f, w0 = P.w0, L = P.len;
        const bool term = P.term != 0, slow = P.slow != 0;
        const long long gbase = base + w0;
        const GAgg &E = P.E;
        // a call sees only its own triggers: "earlier" means earlier in this call
        const long long trig_base = (!BATCH && p.E0) ? p.E0->tdc.n : 0;
        const bool prev_global = E.tdc.n > trig_base;
        TPX_PH(0);

        // ---- read the range, a packet per thread and step, into registers;
        // the TDC packets of each 32 positions are kept as a mask, their
        // words (near a pixel wrap all words) in shared memory ----
        uint64_t w[KM];
#pragma unroll
        for (int j = 0; j < KM; ++j) {
            const int r = j * NTW + tid;
            w[j] = r < L ? __ldcg(p.pk + gbase + r) : 0ull;
        }
        for (int i = tid; i < TW / 4; i += NTW) reinterpret_cast<uint4 *>(S.u1.t.bits)[i] = make_uint4(0, 0, 0, 0);
        for (int i = tid; i < OHB / 2; i += NTW) reinterpret_cast<uint32_t *>(S.u1.t.ohead)[i] = 0xFFFFFFFFu;
#pragma unroll
        for (int j = 0; j < KM; ++j) {
            if (j * NTW >= L) break;
            const int r = j * NTW + tid;
            const bool is_tdc = (w[j] >> 60) == 0x6u;
            const unsigned m = __ballot_sync(0xffffffffu, is_tdc);
            if (lane == 0 && r < L) S.u3.tmask[j * NW + wid] = m;
            if ((is_tdc || slow) && r < L) S.srec[r] = w[j];
        }
        cta_sync();
        TPX_PH(1);

        // ---- the TDC packets before each 32 positions, the positions of all
        // of them, and their unwrapped times (one warp, a scan of the wrap
        // steps) ----
        if (wid == 0) {
            constexpr int GPL = C / 32 / 32;
            const int G = (L + 31) >> 5;
            int c = 0;
#pragma unroll
            for (int k = 0; k < GPL; ++k) {
                const int g = lane * GPL + k;
                c += g < G ? __popc(S.u3.tmask[g]) : 0;
            }
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            const int ntdc = __shfl_sync(0xffffffffu, incl, 31);
            int at = incl - c, mine = 0;
#pragma unroll
            for (int k = 0; k < GPL; ++k) {
                const int g = lane * GPL + k;
                if (g >= G) break;
                S.u4.tpre[g] = (uint16_t)at;
                for (unsigned m = S.u3.tmask[g]; m; m &= m - 1) {
                    const int q = 32 * g + __ffs(m) - 1;
                    if (at < MAXSEG) S.tdc_pos[at] = (uint16_t)q;
                    mine += q < cnt - w0;
                    ++at;
                }
            }
            mine = (int)__reduce_add_sync(0xffffffffu, (unsigned)mine);
            if (lane == 0) {
                S.ntdc = ntdc;
                S.cnt[C_TDCS] = (unsigned long long)mine;   // the tile's own
                if (ntdc > MAXSEG) S.status |= ST_CAPACITY;
                S.tdc_t[min(ntdc, MAXSEG)] = LLONG_MAX;
            }
            const int nseg = min(ntdc, MAXSEG);
            __syncwarp();
            bool has = E.tdc.n > 0;
            long long last = E.tdc.last, ep = E.tdc.sum, t_last = 0;
            for (int i0 = 0; i0 < nseg; i0 += 32) {
                const int i = i0 + lane;
                long long r = 0;
                int q = 0;
                if (i < nseg) {
                    q = S.tdc_pos[i];
                    r = tdc_raw(S.srec[q]);
                }
                const long long rp = __shfl_up_sync(0xffffffffu, r, 1);
                int st = 0;
                if (i < nseg && (lane > 0 || has)) st = (int)jump(r - (lane > 0 ? rp : last), tt);
                int inc = st;
                if (__any_sync(0xffffffffu, st != 0)) {
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int u = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += u;
                    }
                }
                const long long t = r + (ep + inc) * kTdcPeriod;
                const long long tp_ = __shfl_up_sync(0xffffffffu, t, 1);
                if (i < nseg) {
                    S.tdc_t[i] = t;
                    if ((lane > 0 || i0 > 0) && t < (lane > 0 ? tp_ : t_last)) atomicOr(&p.ctl->status, ST_TRIG_ORDER);
                    if (!BATCH && q < cnt - w0) {   // a batch writes its triggers at the flush
                        const long long g = E.tdc.n - trig_base + i;
                        if (g >= 0 && g < p.trig_cap) p.trig[g] = t; else atomicOr(&p.ctl->status, ST_TRIG_CAP);
                    }
                }
                const int lastl = min(31, nseg - 1 - i0);
                ep += __shfl_sync(0xffffffffu, inc, lastl);
                last = __shfl_sync(0xffffffffu, r, lastl);
                t_last = __shfl_sync(0xffffffffu, t, lastl);
                has = true;
            }
        }
        TPX_PH(4);
        if (slow) {
            // a pixel wrap step (Sec. IV.A) lies in or near the range: the
            // wraps of every position, over contiguous chunks of the packets.
            // A thread counts the steps from its first pixel up to the first
            // pixel after its chunk; one scan gives the wraps before each.
            cta_sync();
            const int kpd = (L + NTW - 1) / NTW;
            const int p0 = tid * kpd;
            int fpx = INT_MAX, jp = 0;
            {
                int lpx = -1;
                long long lr = 0;
                for (int q = p0; q < min(p0 + kpd, L); ++q) {
                    const uint64_t v = S.srec[q];
                    if ((v >> 60) != 0xBu) continue;
                    const long long r = pix_raw(v);
                    if (lpx >= 0) jp += (int)jump(r - lr, tp); else fpx = q;
                    lpx = q;
                    lr = r;
                }
                if (lpx >= 0) {   // the step to the next pixel after the chunk
                    for (int q = p0 + kpd; q < L; ++q) {
                        const uint64_t v = S.srec[q];
                        if ((v >> 60) == 0xBu) { jp += (int)jump(pix_raw(v) - lr, tp); break; }
                    }
                }
                const int fw = (int)__reduce_min_sync(0xffffffffu, (unsigned)fpx);
                if (lane == 0 && fw != INT_MAX) atomicMin(&S.first_pix, fw);
            }
            int total;
            const int jp_ex = block_scan_int(S, jp, &total);
            if (tid == 0) {
                const int fp = S.first_pix;
                S.j0 = (fp != INT_MAX && E.pix.n > 0) ? jump(pix_raw(S.srec[fp]) - E.pix.last, tp) : 0;
            }
            cta_sync();
            int d = (int)S.j0 + jp_ex;
            bool any = false;
            long long last = 0;
            for (int q = p0; q < min(p0 + kpd, L); ++q) {
                const uint64_t v = S.srec[q];
                if ((v >> 60) != 0xBu) continue;
                const long long r = pix_raw(v);
                if (any) d += (int)jump(r - last, tp);
                any = true;
                last = r;
                S.spos[q] = (uint16_t)(int16_t)d;
            }
        }
        cta_sync();

        // a batch tile whose range the tiles cannot hold: its run is redone by
        // the general path, so it clusters nothing (its counts still flow).
        // A big range clusters nothing here either: its path runs below.
        const bool big_tile = BIGR && (S.status & ST_BIG) && !(S.status & ST_CAPACITY);
        const int nseg = min(S.ntdc, MAXSEG);
        TPX_PH(3);
        // ---- packets -> shot, cut, timewalk, packed record; each kept pixel
        // takes its bit of the cell table, or a number among those that find
        // it taken ----
        uint32_t rk[(KM + 1) / 2];
#pragma unroll
        for (int j = 0; j < (KM + 1) / 2; ++j) rk[j] = 0u;
        {
            const long long t_prev_global = E.tdc.last + E.tdc.sum * kTdcPeriod;
            const unsigned below = (1u << lane) - 1u;
            unsigned c_pre = 0, c_bg = 0;
            bool exc = false;
#pragma unroll
            for (int j = 0; j < KM; ++j) {
                if (j * NTW >= L || big_tile) { w[j] = INVALID; continue; }
                const int r = j * NTW + tid;
                const uint64_t v = w[j];
                uint64_t rec = INVALID;
                if ((v >> 60) == 0xBu) {   // positions past the range hold zero
                    const int g = j * NW + wid;
                    const int seg = (int)S.u4.tpre[g] + __popc(S.u3.tmask[g] & below) - 1;
                    long long ep = E.pix.sum;
                    if (slow) ep += (int16_t)S.spos[r];
                    const long long t = pix_raw(v) + ep * kPixPeriod;
                    if (seg < 0) {
                        if (!prev_global) ++c_pre;        // no trigger before it anywhere
                    } else if (seg < nseg) {
                        const long long t_lo = S.tdc_t[seg], d = t - t_lo;
                        // the common case: at or after its trigger, before the next one, inside the cut
                        if ((unsigned long long)d <= (unsigned long long)p.tof_max && t < S.tdc_t[seg + 1]) {
                            const int tot = pix_tot(v);
                            const int tofb = (int)d + kTofBias - (p.lut ? (int)p.lut[tot] : 0);
                            rec = mkrec((uint32_t)tofb, (uint32_t)seg, (uint32_t)tot, (uint32_t)pix_x(v), (uint32_t)pix_y(v));
                            const uint32_t b = tbit(rec), m = 1u << (b & 31);
                            if (atomicOr(&S.u1.t.bits[b >> 5], m) & m)
                                rk[j / 2] |= ((uint32_t)atomicAdd(&S.nov, 1) + 1u) << (16 * (j & 1));
                        } else if (t >= S.tdc_t[seg + 1]) {
                            exc = true;                   // after a trigger read out later
                        } else if (d >= 0) {
                            ++c_bg;
                        } else {                          // read out late: an earlier shot's
                            const bool hp = seg > 0 || prev_global;
                            const long long tprev = seg > 0 ? S.tdc_t[seg - 1] : t_prev_global;
                            if (!hp) ++c_pre;
                            else if (t >= tprev && t - tprev > p.tof_max) ++c_bg;
                            else exc = true;
                        }
                    }
                }
                w[j] = rec;
            }
            if (__any_sync(0xffffffffu, (c_pre | c_bg) != 0)) {
                c_pre = __reduce_add_sync(0xffffffffu, c_pre);
                c_bg = __reduce_add_sync(0xffffffffu, c_bg);
                if (lane == 0) { atomicAdd(&S.n_pre, c_pre); atomicAdd(&S.n_bg, c_bg); }
            }
            if (exc) atomicOr(&S.status, ST_EXCEPTION);
        }
        cta_sync();
        TPX_PH(5);

        // ---- the rank of each table word: an exclusive scan of the bit counts ----
        const bool skip = BATCH && (S.status & (ST_CAPACITY | ST_EXCEPTION | ST_BIG)) != 0;
        int nb, nov = S.nov;   // kept pixels in the table, and outside it
        {
            constexpr int WPT = (TW + NTW - 1) / NTW;
            int c[WPT], sum = 0;
#pragma unroll
            for (int k = 0; k < WPT; ++k) {
                c[k] = tid * WPT + k < TW ? __popc(S.u1.t.bits[tid * WPT + k]) : 0;
                sum += c[k];
            }
            int at = block_scan_int(S, sum, &nb);
#pragma unroll
            for (int k = 0; k < WPT; ++k) {
                if (tid * WPT + k < TW) S.u1.t.rank[tid * WPT + k] = (uint16_t)at;
                at += c[k];
            }
            for (int i = tid; i < C / 32; i += NTW) S.u3.rwalk[i] = 0u;
        }
        cta_sync();
        TPX_PH(6);
        // ---- the records into their slots ----
#pragma unroll
        for (int j = 0; j < KM; ++j) {
            if (j * NTW >= L) break;
            const uint64_t rec = w[j];
            if (rec == INVALID) continue;
            const uint32_t b = tbit(rec), o = (rk[j / 2] >> (16 * (j & 1))) & 0xFFFFu;
            const int slot = o ? nb + (int)o - 1 : rank_at(S, b);
            if (!TPX_IN(slot, C)) continue;
            S.srec[slot] = rec;
            S.spos[slot] = (uint16_t)(j * NTW + tid);
            S.par[slot] = (uint16_t)slot;
            S.notpeak[slot] = 0;
            if (o) {   // push it on its chain (16-bit exchange as a CAS loop)
                unsigned short *h = &S.u1.t.ohead[ohash(b)], old = *h, seen;
                do {
                    seen = old;
                    old = atomicCAS(h, seen, (unsigned short)(o - 1));
                } while (old != seen);
                S.u5.onext[o - 1] = old;
            }
        }
        const int kept = nb + nov;
        if (tid < 4) S.srec[kept + tid] = INVALID;   // the probes past the last slot find no cell
        if (skip) nb = nov = 0;
        const int n = nb + nov;
        if (MODE == TPX_MODE_PAPER)   // no union queue: the label entries are free already
            for (int i = tid; i < L; i += NTW) S.u2.lab[i] = NOLAB;
        cta_sync();
        TPX_PH(2);

        // ---- neighbour pass: each adjacent pair of table pixels once (Sec. V.A
        // box rule) ---- A lane's pixel looks at the next slot (its right-hand
        // neighbour, if that is one) and at the slots of the row above, and
        // sets the local-maximum flags (Sec. V.B). CC: the pixel points to one
        // partner (a plain store: pointers only go forward in (y, x), so they
        // form a forest) and queues the pairs that no path of other pairs
        // joins.
        for (int t0 = tid & ~31; t0 < nb; t0 += NTW) {
            const int i = t0 + lane;
            const bool live = i < nb;
            const uint64_t r = live ? S.srec[i] : INVALID;
            const int x = r_x(r), y = r_y(r), tb = r_tof(r), tot = r_tot(r);
            const uint32_t cell = r_cell(r), b = tbit(r);
            bool dim = false;
            if (MODE == TPX_MODE_CC && p.rx == 1 && p.ry == 1) {
                // 8-neighbour box: four probes, no loop. The row above has its
                // (at most three) cells' pixels in consecutive slots from the
                // rank of the first cell on.
                int tmin = INT_MAX, tmax = INT_MIN;
                auto probe = [&](int j, bool ok) -> bool {   // an adjacent pixel: its flags and time
                    const uint64_t rj = S.srec[j];
                    const int tj = r_tof(rj);
                    ok = ok && within(tj - tb, p.dt);
                    if (ok) {
                        if (dimmer(S, i, tot, j, r_tot(rj))) dim = true; else S.notpeak[j] = 1;
                        tmin = min(tmin, tj);
                        tmax = max(tmax, tj);
                    }
                    return ok;
                };
                bool hE = live && i + 1 < nb && x < 255 && r_cell(S.srec[i + 1]) == cell + 1;
                if (hE) hE = probe(i + 1, true);
                int jL = -1, jM = -1, jR = -1;
                if (live && y < 255) {
                    const uint32_t l = x > 0 ? 1u : 0u, span = l + (x < 255 ? 1u : 0u);
                    const int s0 = rank_at(S, (b + 256u) - ((b + 256u) & TB) - l);
                    const uint32_t c0 = cell + 256u - l;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const int j = s0 + k;
                        if (!TPX_IN(j, C + 4)) break;
                        const uint32_t u = r_cell(S.srec[j]) - c0;
                        if (probe(j, u <= span && j < nb)) {
                            const uint32_t v = u + 1u - l;   // 0 left, 1 middle, 2 right
                            if (v == 1) jM = j; else if (v == 0) jL = j; else jR = j;
                        }
                    }
                }
                // Which pairs need a union of their own, when all partners lie
                // within dt of each other (adjacent in time): the pair to the
                // right always (pointer); a pixel above both this pixel and
                // its right-hand neighbour is reached through the neighbour's
                // pair with it (and so on to the right); a diagonal one through
                // the pixel above when there is one. When they do not, every pair.
                const bool close = tmax - tmin <= p.dt || tmin == INT_MAX;
                int up = hE ? i + 1 : jM >= 0 ? jM : jR >= 0 ? jR : jL >= 0 ? jL : i;
                if (close) {
                    if (jL >= 0 && jM < 0 && up != jL) queue_pair(S, i, jL);
                } else {
                    if (jM >= 0 && up != jM) queue_pair(S, i, jM);
                    if (jR >= 0 && up != jR) queue_pair(S, i, jR);
                    if (jL >= 0 && up != jL) queue_pair(S, i, jL);
                }
                // along a row the pointer goes straight to the last slot of
                // the run that this warp sees
                const unsigned run = __ballot_sync(0xffffffffu, hE) & 0x7FFFFFFFu;
                const int len = __ffs(~(run >> lane)) - 1;
                if (len > 0) up = i + len;
                // and from row to row where this warp's slots hold both (the
                // 32 slots span a few rows): three doublings in registers, so
                // that later finds take a hop or two
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int l = up - t0;
                    const int v = __shfl_sync(0xffffffffu, up, l & 31);
                    if ((unsigned)l < 32u) up = v;
                }
                if (live) S.par[i] = (uint16_t)up;
            } else if (live) {
                int up = i;
                bool more = false;
                for (int dy = 0; dy <= p.ry && y + dy <= 255; ++dy) {
                    const int dlo = dy == 0 ? 0 : -min(p.rx, x), dhi = min(p.rx, 255 - x);
                    const uint32_t c0 = cell + (uint32_t)(256 * dy + dlo);
                    int j, s1;
                    row_slots(S, b, dy, dlo, dhi, &j, &s1);
                    for (; j < s1; ++j) {
                        if (j == i || !TPX_IN(j, C)) continue;
                        const uint64_t rj = S.srec[j];
                        if (r_cell(rj) - c0 > (uint32_t)(dhi - dlo) || !within(r_tof(rj) - tb, p.dt)) continue;
                        if (dimmer(S, i, tot, j, r_tot(rj))) dim = true; else S.notpeak[j] = 1;
                        // CC: the pixel points to its first partner; any other is
                        // united in a second walk
                        if (up == i) up = j; else more = true;
                    }
                }
                if (MODE == TPX_MODE_CC) {
                    S.par[i] = (uint16_t)up;
                    if (more) { atomicOr(&S.u3.rwalk[i >> 5], 1u << (i & 31)); S.rw = 1; }
                }
            }
            if (dim) S.notpeak[i] = 1;
        }
        // pixels outside the table: each row of their boxes (dense lanes, the
        // last warps first: they have the fewest slots above). A warp's lanes
        // take one row of consecutive pixels, so that those of a cell hit many
        // times walk its chain together (shots of 500 pixels with 80% of them in
        // one cell, radius 7: 2.50 -> 0.85 ms a call, with the untaken columns
        // left out; with the rows of a pixel on consecutive lanes one lane in
        // 2 ry + 1 walked the chain)
        const int rows = 2 * p.ry + 1;
        for (int t = NTW - 1 - tid; t < nov * rows; t += NTW)
            overflow_row<MODE, false>(S, p, pb, t % nov, t / nov - p.ry, nb);
        cta_sync();
        TPX_PH(7);

        int ncl = 0;
        if (MODE == TPX_MODE_CC) {
            // unions of the queued pairs; the slots marked for a second walk
            // unite each of their partners in turn
            const int nq = min(S.qn, QN);
            for (int k = tid; k < nq; k += NTW) {
                const uint32_t pr = S.u2.queue[k];
                if (TPX_IN(pr >> 16, n) && TPX_IN(pr & 0xFFFFu, n)) uf_unite(pb, pr >> 16, pr & 0xFFFFu);
            }
            if (S.rw)
                for (int i = tid; i < n; i += NTW) {
                    if (!((S.u3.rwalk[i >> 5] >> (i & 31)) & 1u)) continue;
                    if (i < nb) rewalk_unite(S, p, pb, i);
                    else
                        for (int dy = -p.ry; dy <= p.ry; ++dy) overflow_row<MODE, true>(S, p, pb, i - nb, dy, nb);
                }
            cta_sync();
            TPX_PH(9);
            // roots (each slot's pointer is changed by its own thread alone);
            // the cell table is free now: member-list heads, cleared
            for (int i = tid; i < n; i += NTW) {
                uf_st(pb, (uint32_t)i, uf_root(pb, (uint32_t)i));
                S.u1.mhead[i] = EMPTY;
            }
            for (int i = tid; i < C / 32; i += NTW) S.u3.lbits[i] = 0u;
            cta_sync();
            TPX_PH(10);
            // member lists: each kept pixel joins its root's list; the roots
            // are appended to the root list in any order
            for (int t0 = tid & ~31; t0 < n; t0 += NTW) {
                const int i = t0 + lane;
                bool is_root = false;
                if (i < n) {
                    const uint32_t rt = S.par[i];
                    if (TPX_IN(rt, n)) S.u2.mnext[i] = (uint16_t)atomicExch(&S.u1.mhead[rt], (uint32_t)i);
                    is_root = rt == (uint32_t)i;
                }
                const unsigned m = __ballot_sync(0xffffffffu, is_root);
                int at = 0;
                if (lane == 0 && m) at = atomicAdd(&S.nroot, __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (is_root && TPX_IN(at, C)) S.u5.rootpos[at] = (uint16_t)i;
            }
            cta_sync();
            ncl = S.nroot;
        } else {
            // PAPER mode: one record per local maximum, marked by position, and
            // the maxima listed (in the parents' place, which this mode does
            // not use), so that a thread per maximum sums its neighbourhood: one
            // pixel in 24 is one, and a thread per pixel left the other lanes
            // of nearly every warp idle (51% of the kernel; 20,011 shots, radius
            // 2: 1.38 -> 0.88 ms a call)
            for (int i = tid; i < C / 32; i += NTW) S.u3.lbits[i] = 0u;
            cta_sync();
            for (int i0 = wid * 32; i0 < n; i0 += NTW) {
                const int i = i0 + lane;
                const bool pk = i < n && !S.notpeak[i];
                const unsigned m = __ballot_sync(0xffffffffu, pk);
                int at = 0;
                if (lane == 0 && m) at = atomicAdd(&S.nroot, __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (pk && TPX_IN(at, C)) {
                    const uint32_t q = S.spos[i];
                    atomicOr(&S.u3.lbits[q >> 5], 1u << (q & 31));
                    S.par[at] = (uint16_t)i;
                }
            }
            cta_sync();
            ncl = S.nroot;
        }
        bool big_done = false;   // this tile's records wait in the big-range scratch
        if constexpr (BIGR) {
            // a big range takes its own path, once its record slot is free
            if (big_tile) {
                if (tid == 0) wait_count(&S.consumed, ent - NP, p);
                cta_sync();
                const int k = big_range<BATCH>(S, p, gbase, rend, f - w0, C - w0, prev_global, E, ent % NP);
                ncl = k > 0 ? k : 0;
                big_done = k >= 0;
                TPX_PH(17);
            }
        }
        TPX_PH(11);
        // ---- record offsets: publish this tile's count now, look back later ----
        if (tid == 0 && tile + 1 != p.hold) {
            if (tile > 0) {
                __stcg(&p.ts.cagg[tile], (long long)ncl);
                if (BATCH) __stcg(&p.bt.tcagg[tile], (long long)S.cnt[C_TDCS]);
                st_release(&p.ts.cflags[tile], (seq << 2) | 1u);
            } else {
                __stcg(&p.ts.cpre[0], (long long)ncl);
                if (BATCH) __stcg(&p.bt.tcpre[0], (long long)S.cnt[C_TDCS]);
                st_release(&p.ts.cflags[0], (seq << 2) | 2u);
            }
        }
        const long long ntr_here = E.tdc.n - trig_base + (long long)S.cnt[C_TDCS];
        // a tile with nothing to write (no records, no triggers; not a run's
        // first tile nor the call's last) needs no offset: its count is
        // published, and the successors' look-backs add it up
        const bool any = STAGED && (ncl != 0 || S.cnt[C_TDCS] != 0 || (BATCH && tile == tile0) || tile == p.n_tiles - 1);
        // STAGED_ONLY: at the range's position in the stream (the tiles' ranges do
        // not overlap, and a range has no more records than packets), so that the
        // staging holds a call's packets, not a whole range for each of its small
        // tiles (a context of 155,648 packets: 113 -> 38 MB)
        tpx_record *const stage = STAGED_ONLY ? p.stage + gbase
                                  : STAGED ? p.stage + ((long long)blockIdx.x * NP + ent % NP) * C : nullptr;
        if (STAGED) {   // the slot's previous records are out (checked before the next barrier)
            if (tid == 0) wait_count(&S.consumed, ent - NP, p);
        } else if (wid == 0) {   // unstaged: the records' offset now, by an inline look-back
            longlong2 O;
            resolve_offset<false>(p, seq, tile, ncl, ntr_here, 0, 0, false, true, &O);
            if (lane == 0) S.clo = O.x;
        }
        const int ncl_here = big_done ? 0 : ncl;   // records to form here
        auto put = [&](int k, const tpx_record &o) {
            if (STAGED) stage[k] = o;
            else if (k < p.cl_cap - S.clo) out_record(p, S.clo + k, o);
        };
        if (MODE == TPX_MODE_CC) {
            // One thread per cluster walks its member list: the exact integer
            // moments (Sec. V.C) and the cluster's earliest pixel in (time,
            // position) order -- its canonical label -- which is kept in the
            // upper half of the list head and marked in the label bitmap. A
            // thread keeps its first cluster's moments in registers until the
            // labels' ranks are known.
            Moments held{0, 0, 0, 0, 0, 0, 0, 0, 0};
            for (int k = tid; k < ncl_here; k += NTW) {
                if (!TPX_IN(k, C)) break;
                const uint32_t rt = S.u5.rootpos[k];
                if (!TPX_IN(rt, C)) continue;
                const uint32_t head = S.u1.mhead[rt] & 0xFFFFu;
                const Moments m = walk_members(S, p, head);
                if (!TPX_IN(m.best_lo, C)) continue;
                S.u1.mhead[rt] = (m.best_lo << 16) | head;
                atomicOr(&S.u3.lbits[m.best_lo >> 5], 1u << (m.best_lo & 31));
                if (k == tid) held = m;
            }
            cta_sync();
            TPX_PH(12);
            // the labels' ranks: one warp scans the bitmap's counts; the
            // others clear the label entries (they take the member links'
            // place, unless more clusters than threads have to be walked again)
            const bool many = ncl_here > NTW;
            if (wid == 0) scan_label_bits(S);
            else if (!many) for (int q = tid - 32; q < L; q += NTW - 32) S.u2.lab[q] = NOLAB;
            cta_sync();
            TPX_PH(19);
            if (tid < ncl_here && held.n > 0) {
                const int k = label_rank(S, held.best_lo);
                if (TPX_IN(k, C)) put(k, make_record(held, S, p, gbase, E.tdc.n));
            }
            if (many) {
                for (int i = tid + NTW; i < ncl_here; i += NTW) {
                    if (!TPX_IN(i, C)) break;
                    const uint32_t rt = S.u5.rootpos[i];
                    if (!TPX_IN(rt, C)) continue;
                    const Moments m = walk_members(S, p, S.u1.mhead[rt] & 0xFFFFu);
                    const int k = label_rank(S, m.best_lo);
                    if (TPX_IN(k, C)) put(k, make_record(m, S, p, gbase, E.tdc.n));
                }
                cta_sync();
                for (int q = tid; q < L; q += NTW) S.u2.lab[q] = NOLAB;
                cta_sync();
            }
            // the label position of each kept pixel, by position
            if (!big_done) {
                unsigned c = 0;
                for (int i = tid; i < n; i += NTW) {
                    const bool pk = !S.notpeak[i];
                    if (!TPX_IN(S.par[i], C)) continue;
                    S.u2.lab[S.spos[i]] = (uint16_t)((S.u1.mhead[S.par[i]] >> 16) | (pk ? PEAK : 0));
                    c += pk;
                }
                c = __reduce_add_sync(0xffffffffu, c);
                if (lane == 0 && c) atomicAdd(&S.n_pk, c);
            }
        } else {
            if (wid == 0) scan_label_bits(S);
            cta_sync();
            // records: box neighbourhood sums of each local maximum (Sec. V.C)
            for (int i = tid; i < n; i += NTW) {
                const uint32_t q = S.spos[i];
                S.u2.lab[q] = (uint16_t)(q | (S.notpeak[i] ? 0 : PEAK));
            }
            if (tid == 0 && ncl) S.n_pk += (unsigned)ncl;
            for (int at = tid; at < ncl; at += NTW) {
                if (!TPX_IN(at, C)) break;
                const int i = S.par[at];
                const uint32_t q = S.spos[i];
                const uint64_t r = S.srec[i];
                const int x = r_x(r), y = r_y(r), tb = r_tof(r);
                const uint32_t bit = tbit(r), cell = r_cell(r);
                Moments m{0, 0, 0, 0, 0, 1, r_seg(r), q, tb};
                const int dlo = -min(p.rx, x), dhi = min(p.rx, 255 - x);
                for (int dy = -min(p.ry, y); dy <= min(p.ry, 255 - y); ++dy) {
                    const uint32_t c0 = cell + (uint32_t)(256 * dy + dlo);
                    auto add = [&](int j) {
                        const uint64_t rj = S.srec[j];
                        const int tj = r_tof(rj);
                        if (r_cell(rj) - c0 > (uint32_t)(dhi - dlo) || !within(tj - tb, p.dt)) return;
                        const uint32_t aj = (uint32_t)r_tot(rj);
                        m.n += 1;
                        m.s_tot += aj;
                        m.s_x += aj * (uint32_t)r_x(rj);
                        m.s_y += aj * (uint32_t)r_y(rj);
                        m.s_tt += (long long)((uint64_t)aj * (uint32_t)tj);
                        m.tofb0 = min(m.tofb0, tj);
                    };
                    int j, s1;
                    row_slots(S, bit, dy, dlo, dhi, &j, &s1);
                    for (; j < s1; ++j)
                        if (TPX_IN(j, C)) add(j);
                    if (nov == 0) continue;
                    const uint32_t row = (bit + 256u * (uint32_t)dy) & (TB - 1);
                    for (int dx = dlo; dx <= dhi; ++dx)
                        for (uint32_t o = S.u1.t.ohead[ohash(row + dx)]; o != EMPTY; o = S.u5.onext[o]) {
                            if (!TPX_IN(nb + o, C)) break;
                            if (r_cell(S.srec[nb + o]) == cell + (uint32_t)(256 * dy + dx)) add(nb + (int)o);
                        }
                }
                const int k = label_rank(S, q);
                if (TPX_IN(k, C)) put(k, make_record(m, S, p, gbase, E.tdc.n));
            }
        }
        cta_sync();
        TPX_PH(13);
        // ---- per-packet outputs over the range (and the packets before the
        // call's first trigger) ----
        {
            const int W1 = skip ? 0 : (term ? L - 1 : L);
            for (int q = tid; q < W1; q += NTW) {
                if (!TPX_IN(gbase + q, rend)) continue;
                const uint32_t v = S.u2.lab[q];
                const bool k = v != NOLAB;
                const long long lp = (long long)(v & (PEAK - 1));
                if (p.labels) p.labels[gbase + q] = k ? p.idx_base + gbase + lp : -1LL;
                else if (p.labels32) p.labels32[gbase + q] = k ? (int)(p.idx_base - p.lab32_base + gbase + lp) : -1;
                if (p.is_peak) p.is_peak[gbase + q] = k && (v & PEAK) ? 1 : 0;
            }
        }
        TPX_PH(14);
        if (BATCH) {   // this tile's trigger times wait with its records
            const int nt = min((int)S.cnt[C_TDCS], MAXSEG);
            long long *ts = p.bt.tstage + ((long long)blockIdx.x * NP + ent % NP) * T;
            for (int i = tid; i < nt; i += NTW) ts[i] = S.tdc_t[i];
        }
        if (tid == 0) {
            S.cnt[C_PACKETS] = (unsigned long long)cnt;
            S.cnt[C_CLUSTERS] = (unsigned long long)ncl;
            if (!big_done) {   // a big range counted its own pixels
                S.cnt[C_KEPT] = (unsigned long long)kept;
                S.cnt[C_DROP_PRE] = S.n_pre;
                S.cnt[C_DROP_BG] = S.n_bg;
                S.cnt[C_PEAKS] = S.n_pk;
            }
        }
        cta_sync();
        TPX_PH(15);
        // the tile's counters join the CTA's; the tile goes to the service warp
        if (tid == 0) {
            unsigned st = S.status & ~ST_BIG;
            if (BATCH && (st & (ST_CAPACITY | ST_EXCEPTION))) {   // only this run is redone
                p.bt.run_failed[run] = 1u;
                st = (st & ~(ST_CAPACITY | ST_EXCEPTION)) | ST_RUN_REDO;
            }
            if (st) atomicOr(&p.ctl->status, st);
            if (any) {
                Smem::Pend &e = S.pend[ent % NP];
                e.tile = tile;
                if constexpr (STAGED_ONLY) e.at = gbase;
                e.ncl = ncl;
                e.ntr = ntr_here;
                e.ntdc = (int)(ntr_here - (E.tdc.n - trig_base));
                e.run = run;
                e.first = tile == tile0;
                e.big = big_done;
            }
            __threadfence_block();   // the staged records are this CTA's own
            *reinterpret_cast<volatile int *>(&S.entries) = ent + (any ? 1 : 0);
            __threadfence_block();
            *reinterpret_cast<volatile int *>(&S.produced) = it + 1;
        }
        ent += any ? 1 : 0;
        __syncwarp();
        if (tid < C_NUM) {
            S.acc[tid] += S.cnt[tid];
            S.cnt[tid] = 0;
        }
    }
}

int smem_bytes() { return (int)sizeof(Smem); }

// The shared-memory attribute belongs to each device's context: it is set
// once per device (and again on any device beyond the table).
template <int MODE, bool STAGED, bool BATCH>
cudaError_t launch_one(const Params &p, int grid, cudaStream_t s) {
    static std::atomic<bool> attr_done[kAttrDevices];
    const int smem = (int)sizeof(Smem);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < kAttrDevices;
    if (!known || !attr_done[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(fused_kernel<MODE, STAGED, BATCH>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        if (known) attr_done[dev].store(true, std::memory_order_release);
    }
    fused_kernel<MODE, STAGED, BATCH><<<grid, NT, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch(const Params &p, int mode, int grid, cudaStream_t s) {
    const bool cc = mode == TPX_MODE_CC;
    if constexpr (!STAGED_ONLY) {
        if (p.bt.tile_run)   // a batch always stages its output
            return cc ? launch_one<TPX_MODE_CC, true, true>(p, grid, s) : launch_one<TPX_MODE_PAPER, true, true>(p, grid, s);
        if (!p.stage)
            return cc ? launch_one<TPX_MODE_CC, false, false>(p, grid, s) : launch_one<TPX_MODE_PAPER, false, false>(p, grid, s);
    }
    return cc ? launch_one<TPX_MODE_CC, true, false>(p, grid, s) : launch_one<TPX_MODE_PAPER, true, false>(p, grid, s);
}
