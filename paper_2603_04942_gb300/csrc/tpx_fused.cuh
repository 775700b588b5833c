// tpx_fused.cuh -- the fused single-pass TPX3 path for sm_103a.
//
// One persistent kernel reads the packet stream once, after the unwrap
// pre-pass (tpx_prepass.cu), which reads it once before. Each CTA repeatedly
// claims the next tile of T packets (dynamic, in stream order), and:
//   1. owns the laser shots whose TDC packet lies in the tile: its range runs
//      from the tile's first TDC packet to the first one past the tile, both
//      known from the pre-pass's tile table, as is the state of the two ToA
//      unwrap chains (pixels, TDCs; Sec. IV.A) where the range starts;
//   2. reads the range into registers, bins each pixel to the most recent
//      trigger in time, applies the <= tof_max background cut and the optional
//      timewalk table (Sec. IV.B-C);
//   3. puts the kept pixels into the order of a table with one bit per cell
//      (shot, y, x): the neighbours of a pixel are consecutive slots;
//   4. visits each adjacent pair once under the box rule of Sec. V.A; a pair
//      updates the local-maximum flags (Sec. V.B, equal ToT resolved towards
//      the later pixel) and, in CC mode, joins two trees of a lock-free
//      union-find;
//   5. forms exact integer sums per cluster (Sec. V.C), stages the records in
//      label order (the cluster's earliest pixel in (time, position) order),
//      and writes per-packet labels; a warp of its own copies the records out
//      to their offset, a decoupled look-back over the tiles' record counts.
// Pixels whose trigger cannot be decided inside the range, and ranges that
// exceed the on-chip capacities, raise a status bit instead (the kernel never
// traps).  All device waits are bounded.
#pragma once

#include <cstdint>

#include "tpx.h"

namespace tpxk {

constexpr int64_t kPixPeriod = 1LL << 34;
constexpr int64_t kTdcPeriod = 1LL << 36;
constexpr int kTofBias = 32768;            // tof_c + bias >= 1 for int16 timewalk shifts
constexpr int kBatchRing = 4;              // staged tiles per CTA of a batch launch (records, triggers)

// status bits latched in Ctl::status
enum : unsigned {
    ST_CORRUPT = 1u << 0,      // unknown header (reported only when strict)
    ST_TRIG_ORDER = 1u << 1,   // trigger times decrease
    ST_CAPACITY = 1u << 2,     // a range exceeds shared-memory capacity
    ST_EXCEPTION = 1u << 3,    // a pixel's trigger lies outside its range
    ST_CLUSTER_CAP = 1u << 4,  // caller cluster buffer too small
    ST_TRIG_CAP = 1u << 5,     // caller trigger buffer too small
    ST_DEVTIMEOUT = 1u << 6,   // a look-back wait ran out
    ST_RUN_REDO = 1u << 7,     // batch: a run needs the general path (see run_failed)
    ST_BOUNDS = 1u << 8,       // checked build: an index outside its array (the access was skipped)
    ST_BIG = 1u << 9,          // a tile's range exceeds the capacity: the big-range path (never reported)
};

enum CounterIdx {
    C_PACKETS = 0, C_PIXELS, C_TDCS, C_CORRUPT, C_DROP_PRE, C_DROP_BG, C_KEPT, C_CLUSTERS, C_PEAKS,
    C_NUM
};

struct Ctl {                     // per-launch control block, cleared before each launch
    unsigned int tile_counter;
    unsigned int status;
    unsigned long long counters[C_NUM];
    unsigned int prepass_done;   // tiles whose aggregates are written (k_prepass_small)
    unsigned int reserved;
};

// one unwrap chain over a stretch of the stream (64-bit form)
struct GChain { long long n, first, last, sum; };
struct GAgg { GChain pix, tdc; };            // 64 bytes

// what the fused kernel plans a tile's range from: the tile's first TDC packet
// (-1: none), and whether a pixel wrap step lies in the tile or between it and
// the pixel before it
struct TileInfo { int first_tdc, wrap; };

// per-tile records: the unwrap pre-pass's tile aggregates and states, and
// the record-count look-back chain
struct TileScratch {
    GAgg *agg;               // [tiles] unwrap-chain aggregate of each tile
    GAgg *pre;               // [tiles] state before each tile: the TDC chain before the tile, the pixel
                             // chain before the first packet the tile's range reads
    GChain *head;            // [tiles] pixel chain from the tile's start to its first TDC packet
    TileInfo *tinfo;         // [tiles]
    GAgg *blk;               // unwrap_prepass_scratch_bytes(tiles): block totals of the scan
    unsigned int *cflags;    // [tiles] cluster-count chain: (seq<<2)|1 count, |2 inclusive prefix
    long long *cagg;         // [tiles]
    long long *cpre;         // [tiles]
};

// a batch of independent runs in one launch: the tile queue and per-run
// outputs (all device memory)
struct BatchTable {
    const int *tile_run;          // [tiles] run of each tile
    const long long *run_tile0;   // [runs] first tile of each run
    const long long *run_off;     // [runs + 1] packet offsets of the runs
    long long *run_rec_off;       // [runs + 1] out: record offsets
    long long *run_trig_off;      // [runs + 1] out: trigger offsets
    unsigned *run_failed;         // [runs] out: 1 = a range the tiles cannot hold
    long long *tcagg, *tcpre;     // [tiles] trigger-count chain
    long long *tstage;            // [grid * kBatchRing * tile packets] trigger staging
    long long n_runs;
};

struct Params {
    const uint64_t *pk;
    long long n;
    long long idx_base;
    long long *labels;
    int *labels32;            // TPX_FLAG_LABELS32: labels minus lab32_base, as int32 (labels NULL)
    int l2_prefetch;          // the packets are in device memory: prefetch the next tile into L2
    int rec64;                // TPX_FLAG_RECORDS64: clusters holds 64-byte records (no x, y, tof)
    long long lab32_base;
    uint8_t *is_peak;
    tpx_record *clusters;
    long long cl_cap;
    long long *n_clusters;
    long long *trig;
    long long trig_cap;
    long long *n_trig;
    const int16_t *lut;
    int rx, ry, dt, strict;
    long long tof_max;
    long long thr_pix, thr_tdc;
    long long n_tiles;
    unsigned int seq;
    TileScratch ts;
    Ctl *ctl;
    tpx_record *stage;       // per-CTA record staging (range-capacity records per
                             // CTA of the grid, kBatchRing slots of them in a batch,
                             // in label order), or NULL: inline offset look-back
    BatchTable bt;           // batch of runs (tile_run == NULL: one stream)
    long long hold;          // tile + 1 whose look-back flags stay unpublished (0: none): lets a
                             // test run its successors' bounded waits out (TPX_EDEVTIMEOUT)
    unsigned char *big;      // big-range scratch, fused_big_scratch_bytes per CTA of the grid (NULL:
                             // a range past the capacity sends its run to the general path)
    const GAgg *E0;          // unwrap state before the call (NULL: stream start)
    GAgg *state_out;         // state after the call, written by the pre-pass (or NULL)
};

}  // namespace tpxk

// launch entry points (defined in tpx_fused.cu)
namespace tpxk {
// tile geometries of the fused kernel
enum : int { GEO_T4096 = 1, GEO_T2048 = 2, GEO_SMALL = 3 };   // the last for small calls only (tpx_process)
int fused_tile_packets(int geo);
int fused_smem_bytes(int geo);
int fused_threads(int geo);
int fused_range_capacity(int geo);
int fused_ctas_per_sm(int geo);
// global scratch of the big-range path per CTA (batches in CC mode)
size_t fused_big_scratch_bytes(int geo);
// the unwrap pre-pass (tpx_prepass.cu): ts.pre[tile] = the state before each
// tile, *state_out = the state after the call; adds the pixel, TDC and
// corrupt-packet counters. launch_fused runs it before the fused kernel.
size_t unwrap_prepass_scratch_bytes(long long n_tiles);
cudaError_t launch_unwrap_prepass(const Params &p, int T, int grid, cudaStream_t s);
// `mid`, if given, is recorded on `s` between the pre-pass and the fused kernel
cudaError_t launch_fused(const Params &p, int mode, int geo, int grid, cudaStream_t s, cudaEvent_t mid = nullptr);
}  // namespace tpxk
