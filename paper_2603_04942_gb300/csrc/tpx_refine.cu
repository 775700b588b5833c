// tpx_refine.cu -- the learned overlap refiner (not in the paper; its
// multi-hit discussion, Sec. VII.B, motivates it): a cluster larger than a
// few pixels may hold two particles. Its 9x9 patch of ToT and relative ToA
// around the rounded centroid goes through a small multilayer perceptron that
// predicts one or two particles and their positions; below a confidence
// threshold the plain centroid (Sec. V.C) stands.
//
//   patches : clusters with more than `min_pixels` pixels; per packet of such
//             a cluster one cell of its patch (the brighter pixel wins a
//             shared cell, ties to the later one).
//   MLP     : 162 inputs -> H (ReLU) -> H (ReLU) -> 6 outputs: two logits
//             (one / two particles) and two offsets (dx, dy) per particle,
//             in pixels from the patch centre. fp32 tiled GEMMs (a dense
//             contraction), bias/ReLU in the epilogue.
//   training: softmax cross-entropy on the count, squared error on the
//             offsets of the true particles, Adam; one call per minibatch.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "tpx_mlp_train.cuh"
#include "tpx.h"
#include "tpx_common.cuh"
#include "tpx_ctx.h"

namespace tpxr {

using namespace tpxk;

constexpr int PS = 9;                 // patch side
constexpr int PC = PS * PS;           // cells per channel
constexpr int NIN = 2 * PC;           // MLP inputs
constexpr int NOUT = 6;               // logits (2) + offsets (4)

inline bool ck(cudaError_t e, int line = __builtin_LINE()) {
    if (e == cudaSuccess) return false;
    if (std::getenv("TPX_DEBUG")) std::fprintf(stderr, "tpx_refine.cu:%d: %s\n", line, cudaGetErrorString(e));
    return true;
}
inline unsigned grid_for(long long n, int bt = 256) {
    long long g = (n + bt - 1) / bt;
    if (g < 1) g = 1;
    if (g > 152 * 16) g = 152 * 16;
    return (unsigned)g;
}

// ---------------------------------------------------------------- patches
// Which clusters get a patch: counted per block of SELB records, then every
// block places its own behind those of the blocks before it.
constexpr int SELT = 256, SELW = SELT / 32, SELR = 2, SELB = SELT * SELR;
constexpr int PT = 2048, PH = 1024, PTH = 512;   // packets of a tile, of its margins; threads of k_patch_tiles
struct TileSel { unsigned first_inv, count; };   // the selected clusters whose root lies in a tile: 2^32 - 1 - the first, how many
struct SelRoot { long long root, raw0; unsigned n; short cx, cy; };   // what k_patch_tiles needs of a selected cluster, in one load
struct PatchInfo {               // read back once per call
    unsigned long long n_sel;    // selected clusters
    unsigned n_inc;              // patches not completed by the tiles (listed)
    unsigned n_far;              // of those, the ones that the wider search could not complete either
    unsigned odd;                // labels not strictly ascending, or outside the packets, or a centre off the sensor: no tiles
    unsigned reserved;
};
// The wider search reads 262 KB of labels a patch (55 ns), the kernels that look
// anywhere all of them once (3.9 us per 10^6 packets, and 15 us of launches).
__host__ __device__ inline bool search_wider(unsigned n_inc, long long n) {
    return (unsigned long long)n_inc << 14 <= (unsigned long long)n + (1ull << 22);
}
__device__ __forceinline__ unsigned sel_flags(const tpx_record *cl, long long ncl, int min_px, unsigned (&m)[SELR],
                                              unsigned *s_c, unsigned *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned c = 0;
#pragma unroll
    for (int j = 0; j < SELR; ++j) {
        const long long i = blockIdx.x * (long long)SELB + w * (32 * SELR) + 32 * j + lane;
        m[j] = __ballot_sync(0xffffffffu, i < ncl && cl[i].n > min_px);
        c += __popc(m[j]);
    }
    if (lane == 0) s_c[w] = c;
    __syncthreads();
    unsigned before = 0, all = 0;
#pragma unroll
    for (int k = 0; k < SELW; ++k) {
        before += k < w ? s_c[k] : 0u;
        all += s_c[k];
    }
    *total = all;
    return before;
}
__global__ void __launch_bounds__(SELT) k_sel_count(const tpx_record *cl, long long ncl, int min_px, unsigned *bcnt) {
    __shared__ unsigned s_c[SELW];
    unsigned m[SELR], total;
    (void)sel_flags(cl, ncl, min_px, m, s_c, &total);
    if (threadIdx.x == 0) bcnt[blockIdx.x] = total;
}
// every block's first slot, beyond kResumBlocks blocks (one block)
constexpr long long kResumBlocks = 4096;
__global__ void __launch_bounds__(1024) k_sel_scan(unsigned *bcnt, long long nb) {
    __shared__ unsigned s[1024];
    unsigned carry = 0;
    for (long long b0 = 0; b0 < nb; b0 += 1024) {
        const long long b = b0 + threadIdx.x;
        const unsigned v = b < nb ? bcnt[b] : 0u;
        s[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {
            const unsigned u = threadIdx.x >= o ? s[threadIdx.x - o] : 0u;
            __syncthreads();
            s[threadIdx.x] += u;
            __syncthreads();
        }
        if (b < nb) bcnt[b] = carry + s[threadIdx.x] - v;
        carry += s[1023];
        __syncthreads();
    }
}
__global__ void __launch_bounds__(SELT) k_select(const uint64_t *pk, const tpx_record *cl, long long ncl, int min_px,
                                                 const unsigned *bcnt, long long nb, long long cap, long long base,
                                                 long long n, long long *sel, int *centre, long long *n_patches,
                                                 TileSel *tiles, SelRoot *roots, PatchInfo *info) {
    __shared__ unsigned s_c[SELW];
    __shared__ unsigned s_sum[SELW];
    unsigned m[SELR], total;
    unsigned o = sel_flags(cl, ncl, min_px, m, s_c, &total);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned first = 0;
    if (nb > kResumBlocks) first = bcnt[blockIdx.x];
    else {
        unsigned v = 0;
        for (unsigned k = threadIdx.x; k < blockIdx.x; k += SELT) v += bcnt[k];
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) s_sum[w] = v;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < SELW; ++k) first += s_sum[k];
    }
#pragma unroll
    for (int j = 0; j < SELR; ++j) {
        const long long i = blockIdx.x * (long long)SELB + w * (32 * SELR) + 32 * j + lane;
        const long long s = (long long)first + o + __popc(m[j] & ((1u << lane) - 1u));
        o += __popc(m[j]);
        const long long label = i < ncl ? cl[i].label : 0, r = label - base;
        if (i < ncl && i > 0 && cl[i - 1].label >= label) info->odd = 1u;
        const bool mine = (m[j] >> lane) & 1u, in = r >= 0 && r < n;
        if (mine && !in) info->odd = 1u;
        // the tile's count and first slot, once per warp and tile: the warp's
        // slots follow one another, and so do their tiles
        const unsigned put = __ballot_sync(0xffffffffu, mine && in && s < cap);
        if ((put >> lane) & 1u) {
            const unsigned tile = (unsigned)(r / PT), peers = __match_any_sync(put, tile);
            if (lane == __ffs(peers) - 1) {
                atomicMax(&tiles[tile].first_inv, 0xFFFFFFFFu - (unsigned)s);
                atomicAdd(&tiles[tile].count, (unsigned)__popc(peers));
            }
        }
        if (!mine || s >= cap) continue;
        const tpx_record &c = cl[i];
        sel[s] = i;
        int cx = 0, cy = 0;
        if (c.s_tot > 0) {   // the centroid rounded half up, exactly: floor((2 s_x + s_tot) / (2 s_tot))
            const long long d = 2 * c.s_tot, nx = 2 * c.s_x + c.s_tot, ny = 2 * c.s_y + c.s_tot;
            if (((unsigned long long)nx | (unsigned long long)ny | (unsigned long long)d) >> 32) {
                cx = (int)(nx / d);
                cy = (int)(ny / d);
            } else {   // the usual cluster: 32-bit divisions
                cx = (int)((unsigned)nx / (unsigned)d);
                cy = (int)((unsigned)ny / (unsigned)d);
            }
        } else if (r >= 0 && r < n) {   // no charge: the earliest pixel
            cx = pix_x(pk[r]);
            cy = pix_y(pk[r]);
        }
        centre[2 * s] = cx;
        centre[2 * s + 1] = cy;
        if ((unsigned)cx > 255u || (unsigned)cy > 255u) info->odd = 1u;
        SelRoot v;
        v.root = r;
        v.raw0 = r >= 0 && r < n ? pix_raw(pk[r]) : 0;
        v.n = (unsigned)c.n;
        v.cx = (short)cx;   // within the sensor, or the call is odd
        v.cy = (short)cy;
        roots[s] = v;
    }
    if (blockIdx.x == nb - 1 && threadIdx.x == 0) {
        *n_patches = (long long)first + total;
        info->n_sel = (unsigned long long)first + total;
    }
}

// a pixel's two patch values. Channel 0: ToT / 1023 rounded to bf16; channel 1:
// ToA relative to the cluster's earliest pixel, in units of 32 ticks (50 ns),
// clamped to [-8, 8], rounded to fp16 (exact: multiples of 1/32 below 8); both
// are exact in bf16 as well
// (the product with the rounded 1 / 1023 rounds to the same bf16 as the quotient
// for all 1024 ToT values)
__device__ __forceinline__ float patch_tot(int tot) { return __bfloat162float(__float2bfloat16_rn((float)tot * (1.f / 1023.f))); }
// (the ticks already clamped to 256 = 8 units either way)
__device__ __forceinline__ float patch_rel(int ticks) { return __half2float(__float2half_rn((float)ticks * 0.03125f)); }
// elements e and e + 1 of a patch row
// (one store where the caller's buffer is aligned to the pair)
__device__ __forceinline__ void put_pair(float *row, int e, float a, float b) {
    if (reinterpret_cast<uintptr_t>(row) & 7) {
        row[e] = a;
        row[e + 1] = b;
    } else {
        *reinterpret_cast<float2 *>(row + e) = make_float2(a, b);
    }
}
__device__ __forceinline__ void put_pair(uint16_t *row, int e, float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    if (reinterpret_cast<uintptr_t>(row) & 3) {
        reinterpret_cast<__nv_bfloat16 *>(row)[e] = v.x;
        reinterpret_cast<__nv_bfloat16 *>(row)[e + 1] = v.y;
    } else {
        *reinterpret_cast<__nv_bfloat162 *>(row + e) = v;
    }
}

// A cluster's packets lie close to one another in the stream (within its shot's
// readout), so a CTA takes the clusters whose earliest pixel is among PT
// packets, with their cells in shared memory, and looks for their members
// there and in PH packets on either side; a patch whose members all turned up
// (the record's count) is written at once, the others are listed for the
// kernels below. Where the shots are so long that more than half of the patches
// before a tile's have gone on (by when it starts), the tile hands its own on
// untried: a patch is the same by any way, and the tiles' way and then the last
// kernels' costs 11 + 4 + 25 f us per 10^6 packets with a share f of them going
// on, the last kernels alone 27. A cell's word holds all that its values follow
// from: ToT, the packet's place in the window (the brighter pixel wins, ties go
// to the later) and the clamped time, never zero. Bound by instruction issue
// (77% of the slots) and by the latency of its steps, so every thread's loads of
// a step are in flight together; the bytes are the labels (twice, half of them
// from L2) and the patches, 31% of the copy rate. In the last kernels every cell has an
// 8-byte key in global memory, cleared, updated and read back, as all of them
// had before: 300 us of the 460 of a call of 440,000 patches of 20 particles a
// shot, now about 115 of 280.
constexpr int PMAX = 96;                         // clusters a pass holds (2048 packets of 24-pixel clusters: 85)
constexpr int PWIN = PT + 2 * PH, PU = PWIN / PTH;
static_assert(PWIN <= 4096, "the window position has 12 bits");
constexpr int kRelMax = 256;                     // 8 units of 32 ticks
__device__ __forceinline__ int rel_ticks(long long raw, long long raw0) {
    long long d = (raw - raw0) & (kPixPeriod - 1);
    if (d >= kPixPeriod / 2) d -= kPixPeriod;   // the signed difference, wrap-safe
    return (int)min((long long)kRelMax, max(-(long long)kRelMax, d));
}
__device__ __forceinline__ unsigned cell_word(int tot, unsigned at, int rel) {
    return ((unsigned)tot << 22) | (at << 10) | (unsigned)(rel + kRelMax + 1);
}
template <typename OutT>
__device__ __forceinline__ void write_patch(OutT *row, const unsigned *key, int lane) {
#pragma unroll
    for (int e = 2 * lane; e < NIN; e += 64) {
        float v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool t = e + u < PC;
            const unsigned x = key[t ? e + u : e + u - PC];
            v[u] = x == 0u ? 0.f : t ? patch_tot((int)(x >> 22)) : patch_rel((int)(x & 1023u) - kRelMax - 1);
        }
        put_pair(row, e, v[0], v[1]);
    }
}
// one warp: lists those of the patches p0 .. p0 + m that go on
template <class F>
__device__ __forceinline__ void list_patches(int m, F goes_on, unsigned p0, unsigned *inc, PatchInfo *info) {
    const int lane = threadIdx.x & 31;
    unsigned f[PMAX / 32], cnt = 0, at = 0;
#pragma unroll
    for (int u = 0; u < PMAX / 32; ++u) {
        f[u] = __ballot_sync(0xffffffffu, 32 * u + lane < m && goes_on(32 * u + lane));
        cnt += __popc(f[u]);
    }
    if (cnt == 0) return;
    if (lane == 0) at = atomicAdd(&info->n_inc, cnt);
    at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
    for (int u = 0; u < PMAX / 32; ++u) {
        if ((f[u] >> lane) & 1u) inc[at + __popc(f[u] & ((1u << lane) - 1u))] = p0 + 32 * u + lane;
        at += __popc(f[u]);
    }
}
template <typename OutT>
__global__ void __launch_bounds__(PTH, 4) k_patch_tiles(const uint64_t *pk, long long n, long long base,
                                                        const long long *labels, const SelRoot *roots,
                                                        const TileSel *tiles, OutT *patch, unsigned *inc,
                                                        PatchInfo *info) {
    __shared__ unsigned s_key[PMAX * PC];
    __shared__ __align__(4) unsigned char s_slot[PT];   // of each packet of the tile: its cluster's place in this pass + 1
    __shared__ int s_c[PMAX];                           // the centre, x | y << 16
    __shared__ unsigned s_cnt[PMAX], s_n[PMAX];
    __shared__ long long s_raw0[PMAX];
    static_assert(PMAX < 255 && PMAX % 32 == 0 && sizeof(s_key) + PT + 24 * PMAX < 48 * 1024, "shared memory of a pass");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long a = blockIdx.x * (long long)PT, w0 = a - PH;
    const int tile_n = (int)min((long long)PT, n - a);
    // the selected clusters of the tile: labels ascend, so they are consecutive
    const TileSel ts = tiles[blockIdx.x];
    const unsigned odd = info->odd;
    const unsigned gone = threadIdx.x == 0 ? __ldcg(&info->n_inc) : 0u;
    if (!ts.count || odd) return;
    const unsigned s0 = 0xFFFFFFFFu - ts.first_inv, s1 = s0 + ts.count;
    if (__syncthreads_or(gone > 2048u && gone > s0 / 2)) {
        if (warp == 0)
            for (unsigned p0 = s0; p0 < s1; p0 += PMAX)
                list_patches((int)min((unsigned)PMAX, s1 - p0), [](int) { return true; }, p0, inc, info);
        return;
    }
    auto root_of = [&](unsigned p0, int m) -> SelRoot { return threadIdx.x < m ? roots[p0 + threadIdx.x] : SelRoot{}; };
    auto clear = [&](int m) {
        for (int k = threadIdx.x; k < PT / 4; k += PTH) reinterpret_cast<unsigned *>(s_slot)[k] = 0u;
        for (int k = threadIdx.x; k < m * PC; k += PTH) s_key[k] = 0u;
    };
    int m = (int)min((unsigned)PMAX, ts.count);
    SelRoot v = root_of(s0, m);
    clear(m);
    int L[PU];
#pragma unroll
    for (int u = 0; u < PU; ++u) {
        const long long q = w0 + u * PTH + threadIdx.x;
        const long long lab = q >= 0 && q < n ? labels[q] : -1ll;
        const unsigned long long r = (unsigned long long)(lab - base - a);
        L[u] = lab >= 0 && r < (unsigned)tile_n ? (int)r : -1;
    }
    for (unsigned p0 = s0;;) {
        __syncthreads();
        if (threadIdx.x < m) {
            s_slot[v.root - a] = (unsigned char)(threadIdx.x + 1);
            s_n[threadIdx.x] = v.n;
            s_raw0[threadIdx.x] = v.raw0;
            s_c[threadIdx.x] = (int)(unsigned short)v.cx | ((int)v.cy << 16);
            s_cnt[threadIdx.x] = 0u;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < PU; h += PU / 2) {   // half of the window's packets in flight together
            int k[PU / 2];
            uint64_t w[PU / 2];
#pragma unroll
            for (int u = 0; u < PU / 2; ++u) {
                k[u] = L[h + u] >= 0 ? (int)s_slot[L[h + u]] - 1 : -1;
                w[u] = k[u] >= 0 ? pk[w0 + (h + u) * PTH + threadIdx.x] : 0ull;
            }
#pragma unroll
            for (int u = 0; u < PU / 2; ++u) {
                if (k[u] < 0) continue;
                atomicAdd(&s_cnt[k[u]], 1u);
                const int c = s_c[k[u]];
                const int dx = pix_x(w[u]) - (c & 0xFFFF) + PS / 2, dy = pix_y(w[u]) - (c >> 16) + PS / 2;
                if (dx < 0 || dx >= PS || dy < 0 || dy >= PS) continue;
                atomicMax(&s_key[k[u] * PC + dy * PS + dx],
                          cell_word(pix_tot(w[u]), (unsigned)((h + u) * PTH + threadIdx.x), rel_ticks(pix_raw(w[u]), s_raw0[k[u]])));
            }
        }
        __syncthreads();
        if (warp == PTH / 32 - 1) list_patches(m, [&](int j) { return s_cnt[j] != s_n[j]; }, p0, inc, info);
        for (int j = warp; j < m; j += PTH / 32)
            if (s_cnt[j] == s_n[j]) write_patch(patch + (p0 + j) * (long long)NIN, s_key + j * PC, lane);
        p0 += PMAX;
        if (p0 >= s1) break;
        m = (int)min((unsigned)PMAX, s1 - p0);
        v = root_of(p0, m);
        __syncthreads();
        clear(m);
    }
}

// The listed patches, when they are few, with a wider search, a CTA each: PW
// packets on either side of the root. (Of 25 particles a shot one in a few
// thousand leaves the window, of 110 one in four.) What is still incomplete goes
// on to the second list. Tried: a CTA for all listed patches of a tile, going on
// from its window until every member turned up; it costs 15 us per 10^6 packets
// at 110 particles a shot and 43 at 500, more than the last kernels.
constexpr int PW = 16384, PWT = 256;
template <typename OutT>
__global__ void __launch_bounds__(PWT) k_patch_wide(const uint64_t *pk, long long n, long long base, const long long *labels,
                                                    const tpx_record *cl, const long long *sel, const int *centre,
                                                    const unsigned *inc, OutT *patch, unsigned *far, PatchInfo *info) {
    __shared__ unsigned long long s_key[PC];     // ToT + 1, place in the window, time (as cell_word, more bits)
    __shared__ unsigned s_word[PC];
    __shared__ unsigned s_cnt;
    const unsigned ni = info->n_inc;
    if (!search_wider(ni, n)) return;
    for (unsigned j = blockIdx.x; j < ni; j += gridDim.x) {
        const long long s = inc[j];
        const tpx_record &c = cl[sel[s]];
        const long long root = c.label - base, w0 = max(0ll, root - PW), w1 = min(n, root + PW);
        const long long raw0 = pix_raw(pk[root]);
        const int cx = centre[2 * s], cy = centre[2 * s + 1];
        __syncthreads();
        if (threadIdx.x < PC) s_key[threadIdx.x] = 0ull;
        if (threadIdx.x == 0) s_cnt = 0u;
        __syncthreads();
#pragma unroll 8
        for (long long q = w0 + threadIdx.x; q < w1; q += PWT) {
            if (labels[q] != c.label || c.label < 0) continue;   // (below 0: no cluster's, as in the tiles)
            atomicAdd(&s_cnt, 1u);
            const uint64_t w = pk[q];
            const int dx = pix_x(w) - cx + PS / 2, dy = pix_y(w) - cy + PS / 2;
            if (dx < 0 || dx >= PS || dy < 0 || dy >= PS) continue;
            atomicMax(&s_key[dy * PS + dx], ((unsigned long long)pix_tot(w) << 42) | ((unsigned long long)(q - w0) << 10) |
                                                (unsigned long long)(rel_ticks(pix_raw(w), raw0) + kRelMax + 1));
        }
        __syncthreads();
        if (s_cnt != (unsigned)c.n) {
            if (threadIdx.x == 0) far[atomicAdd(&info->n_far, 1u)] = (unsigned)s;
            continue;
        }
        if (threadIdx.x < PC) {
            const unsigned long long x = s_key[threadIdx.x];
            s_word[threadIdx.x] = (unsigned)(x >> 42 << 22) | (unsigned)(x & 1023u);
        }
        __syncthreads();
        if (threadIdx.x < 32) write_patch(patch + s * (long long)NIN, s_word, (int)threadIdx.x);
    }
}

// ---- patches the tiles could not complete: member packets anywhere ----
// the list of all patches (odd calls)
__global__ void k_list_all(unsigned *inc, long long ns) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ns; i += (long long)gridDim.x * blockDim.x) inc[i] = (unsigned)i;
}
// the listed patch of each root packet
__global__ void k_roots(const SelRoot *roots, const unsigned *list, long long ni, long long n, int *slot_of_root) {
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < ni; j += (long long)gridDim.x * blockDim.x) {
        const long long r = roots[list[j]].root;
        if (r >= 0 && r < n) slot_of_root[r] = (int)j;   // else not a record of these packets: an empty patch
    }
}
// no root is listed, no cell hit
__global__ void k_clear(int *slot_of_root, long long n, unsigned long long *key, long long cells) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < max(n, cells); i += (long long)gridDim.x * blockDim.x) {
        if (i < n) slot_of_root[i] = -1;
        if (i < cells) key[i] = 0ull;
    }
}
// The brighter pixel of a shared cell wins (ties: the later one). As cell_word,
// the key holds all that the cell's values follow from, the packet's place in 40
// bits: the patches are then written from the keys alone (631,000 patches: 246
// -> 134 us, against reading the winner's packet again for every cell).
__global__ void k_patch_keys(const uint64_t *pk, long long n, long long base, const long long *labels,
                             const int *slot_of_root, const unsigned *list, const SelRoot *roots, const int *centre,
                             unsigned long long *key) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const long long L = labels[q] - base;
        if (labels[q] < 0 || L < 0 || L >= n) continue;
        const int j = slot_of_root[L];
        if (j < 0) continue;
        const unsigned s = list[j];
        const SelRoot v = roots[s];
        const int cx = centre ? centre[2ll * s] : v.cx, cy = centre ? centre[2ll * s + 1] : v.cy;
        const uint64_t w = pk[q];
        const int dx = pix_x(w) - cx + PS / 2, dy = pix_y(w) - cy + PS / 2;
        if (dx < 0 || dx >= PS || dy < 0 || dy >= PS) continue;
        atomicMax(&key[(long long)j * PC + dy * PS + dx], ((unsigned long long)(pix_tot(w) + 1) << 50) | ((unsigned long long)q << 10) |
                                                              (unsigned long long)(rel_ticks(pix_raw(w), v.raw0) + kRelMax + 1));
    }
}
// a thread per cell; empty cells 0
template <typename OutT>
__global__ void k_patch_fill(const unsigned *list, const unsigned long long *key, long long ni, OutT *patch) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ni * PC; c += (long long)gridDim.x * blockDim.x) {
        const long long j = c / PC;
        const unsigned long long k = key[c];
        const float tot = k ? patch_tot((int)(k >> 50) - 1) : 0.f, rel = k ? patch_rel((int)(k & 1023u) - kRelMax - 1) : 0.f;
        OutT *row = patch + list[j] * (long long)NIN + (c - j * PC);
        if constexpr (sizeof(OutT) == 4) {
            row[0] = tot;
            row[PC] = rel;
        } else {
            reinterpret_cast<__nv_bfloat16 *>(row)[0] = __float2bfloat16_rn(tot);
            reinterpret_cast<__nv_bfloat16 *>(row)[PC] = __float2bfloat16_rn(rel);
        }
    }
}

// ---------------------------------------------------------------- GEMM
// C[M x N] = op(A)[M x K] * op(B)[K x N] (+ bias[N]) (ReLU), with op given
// by strides: A(i, k) = A[i * sam + k * sak], B(k, j) = B[k * sbk + j * sbn].
// 64 x 64 tiles, 256 threads, 4 x 4 outputs per thread.
constexpr int TM = 64, TN = 64, TK = 16;
__global__ void __launch_bounds__(256) k_gemm(const float *A, long long sam, long long sak, const float *B,
                                              long long sbk, long long sbn, float *C, long long ldc, int M, int N,
                                              int K, const float *bias, int relu, int accumulate) {
    __shared__ float As[TK][TM + 4];
    __shared__ float Bs[TK][TN + 4];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < K; k0 += TK) {
        // consecutive threads walk the operand's unit-stride dimension (coalesced loads)
        for (int t = threadIdx.x; t < TK * TM; t += 256) {
            const int kk = sak == 1 ? t % TK : t / TM, ii = sak == 1 ? t / TK : t % TM;
            const int i = i0 + ii, k = k0 + kk;
            As[kk][ii] = (i < M && k < K) ? A[i * sam + k * sak] : 0.f;
        }
        for (int t = threadIdx.x; t < TK * TN; t += 256) {
            const int kk = sbk == 1 ? t % TK : t / TN, jj = sbk == 1 ? t / TK : t % TN;
            const int j = j0 + jj, k = k0 + kk;
            Bs[kk][jj] = (j < N && k < K) ? B[k * sbk + j * sbn] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[kk][ty * 4 + r];
#pragma unroll
            for (int r = 0; r < 4; ++r) b[r] = Bs[kk][tx * 4 + r];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(a[r], b[q], acc[r][q]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + ty * 4 + r, j = j0 + tx * 4 + q;
            if (i >= M || j >= N) continue;
            float v = acc[r][q];
            if (accumulate) v += C[(long long)i * ldc + j];
            if (bias) v += bias[j];
            if (relu) v = fmaxf(v, 0.f);
            C[(long long)i * ldc + j] = v;
        }
}
void gemm(cudaStream_t s, const float *A, long long sam, long long sak, const float *B, long long sbk, long long sbn,
          float *C, long long ldc, int M, int N, int K, const float *bias, bool relu, bool accumulate = false) {
    dim3 g((N + TN - 1) / TN, (M + TM - 1) / TM);
    k_gemm<<<g, 256, 0, s>>>(A, sam, sak, B, sbk, sbn, C, ldc, M, N, K, bias, relu ? 1 : 0, accumulate ? 1 : 0);
}

// parameter layout (floats): W1[NIN x H], b1[H], W2[H x H], b2[H], W3[H x NOUT], b3[NOUT]
struct Layout {
    int h;
    long long w1, b1, w2, b2, w3, b3, total;
    __host__ __device__ explicit Layout(int hidden) : h(hidden) {
        w1 = 0; b1 = w1 + (long long)NIN * h; w2 = b1 + h; b2 = w2 + (long long)h * h; w3 = b2 + h;
        b3 = w3 + (long long)h * NOUT; total = b3 + NOUT;
    }
};

// loss of a minibatch and its gradient at the outputs: y = [count(1|2), dx1, dy1, dx2, dy2]
__global__ void k_loss(const float *out, const float *y, int n, float w_off, float *dout, float *loss) {
    __shared__ float part[256];
    float l = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float *o = out + (long long)i * NOUT;
        const float *t = y + (long long)i * 5;
        const int two = t[0] > 1.5f;
        const float m = fmaxf(o[0], o[1]);
        const float e0 = __expf(o[0] - m), e1 = __expf(o[1] - m), z = e0 + e1;
        const float p1 = e1 / z;
        l += -((two ? o[1] : o[0]) - m - __logf(z));
        float *g = dout + (long long)i * NOUT;
        const float inv = 1.f / (float)n;
        g[0] = ((1.f - p1) - (two ? 0.f : 1.f)) * inv;
        g[1] = (p1 - (two ? 1.f : 0.f)) * inv;
        for (int k = 0; k < 4; ++k) {
            const bool used = k < 2 || two;
            const float d = used ? o[2 + k] - t[1 + k] : 0.f;
            l += 0.5f * w_off * d * d;
            g[2 + k] = w_off * d * inv;
        }
    }
    part[threadIdx.x] = l;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, part[0] / (float)n);
}
// dZ = dA where the forward activation was positive (ReLU)
__global__ void k_relu_back(float *d, const float *act, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        if (act[i] <= 0.f) d[i] = 0.f;
}
// bias gradient: column sums of dZ [n x m]
__global__ void k_colsum(const float *d, int n, int m, float *g) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < m; j += gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int i = 0; i < n; ++i) s += d[(long long)i * m + j];
        g[j] = s;
    }
}
__global__ void k_adam(float *p, const float *g, float *m, float *v, long long n, float lr, float b1, float b2,
                       float c1, float c2, float eps) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi, vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// refined hits: per patch the network's two positions when it is confident of
// two particles, else the plain centroid (k = 1 when it is confident of one,
// k = 0 when of neither). p(two) >= thr  <=>  logit margin o1 - o0 >= log(thr / (1 - thr)),
// decided on the fp32 margin so the count is exact, not at the mercy of exp.
__global__ void k_decide(const float *out, const tpx_record *cl, const long long *sel, const int *centre, long long n,
                         float lt, float *hits /* n x 5: n_hits, x1, y1, x2, y2 */) {
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const float *o = out + s * NOUT;
        const float margin = o[1] - o[0];
        const float cx = (float)centre[2 * s], cy = (float)centre[2 * s + 1];
        float *h = hits + s * 5;
        if (margin >= lt) {   // two particles: the network's positions
            h[0] = 2.f; h[1] = cx + o[2]; h[2] = cy + o[3]; h[3] = cx + o[4]; h[4] = cy + o[5];
        } else {              // one particle (1), or not confident (0): the plain centroid
            const tpx_record &r = cl[sel[s]];
            h[0] = -margin >= lt ? 1.f : 0.f; h[1] = (float)r.x; h[2] = (float)r.y; h[3] = 0.f; h[4] = 0.f;
        }
    }
}

// ---------------------------------------------------------------- bf16 inference
// The whole network in one persistent kernel on the tensor cores
// (mma.sync m16n8k16, bf16 operands, fp32 accumulation). Each warp owns 16 MT
// patches and carries them through the three layers: the fp32 accumulator
// fragment of one layer, after bias and ReLU, is exactly the bf16 A-operand
// fragment of the next (row g = lane / 4 and column pair 2 (lane % 4) of
// n-tile j are row g, k pair of k-step j / 2), so activations never leave
// registers. The weights, transposed to [n][k] bf16 by tpx_refiner_pack, sit
// in shared memory for the kernel's lifetime; patches stream from global
// memory as fp32 pairs (8-byte loads; a row's 4 lanes read one 32-byte
// sector) and are rounded to bf16 (exact for the patch precisions).
constexpr int K1P = 176;                       // 162 inputs padded to 11 k-steps
constexpr int S1 = K1P + 8;                    // smem row stride of W1t (92 words: conflict-free)
template <int H> struct MlpGeo {
    static constexpr int S2 = H + 8;           // smem row stride of W2t / W3t
    static constexpr int NT = H / 8;           // n-tiles of a hidden layer
    static constexpr int KS = H / 16;          // k-steps over a hidden layer
    static constexpr size_t w1 = 0, w2 = w1 + (size_t)H * K1P, w3 = w2 + (size_t)H * H, wend = w3 + (size_t)8 * H;
    static constexpr size_t packed_bytes = ((wend * 2 + 15) / 16) * 16 + (size_t)(2 * H + 8) * 4;
    static constexpr size_t smem = (size_t)H * S1 * 2 + (size_t)H * S2 * 2 + (size_t)8 * S2 * 2 + (size_t)(2 * H + 8) * 4;
};
inline size_t packed_bias_off(size_t wend) { return ((wend * 2 + 15) / 16) * 16; }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);   // .x (lower k) in the low half
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// fp32 parameters -> W1t [H][176], W2t [H][H], W3t [8][H] bf16 (zero padded),
// then b1, b2, b3 (padded to 8) fp32
template <int H>
__global__ void k_pack(const float *P, uint16_t *wt, float *bias) {
    using G = MlpGeo<H>;
    const Layout L(H);
    const long long total = (long long)G::wend + 2 * H + 8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        if (i >= (long long)G::wend) {
            const int b = (int)(i - G::wend);
            bias[b] = b < H ? P[L.b1 + b] : b < 2 * H ? P[L.b2 + b - H] : (b - 2 * H < NOUT ? P[L.b3 + b - 2 * H] : 0.f);
            continue;
        }
        float v = 0.f;
        if (i < (long long)G::w2) {
            const int j = (int)(i / K1P), k = (int)(i % K1P);
            if (k < NIN) v = P[L.w1 + (long long)k * H + j];
        } else if (i < (long long)G::w3) {
            const long long r = i - G::w2;
            const int j = (int)(r / H), k = (int)(r % H);
            v = P[L.w2 + (long long)k * H + j];
        } else {
            const long long r = i - G::w3;
            const int j = (int)(r / H), k = (int)(r % H);
            if (j < NOUT) v = P[L.w3 + (long long)k * NOUT + j];
        }
        __nv_bfloat16 b = __float2bfloat16_rn(v);
        wt[i] = *reinterpret_cast<uint16_t *>(&b);
    }
}

// hidden layer epilogue: bias was the accumulator's start; ReLU, round to
// bf16 and regroup n-tile pairs into next-layer A fragments
template <int NT>
__device__ __forceinline__ void to_frags(const float (&acc)[NT][4], uint32_t (&a)[NT / 2][4]) {
#pragma unroll
    for (int s = 0; s < NT / 2; ++s) {
        a[s][0] = pack_bf16(fmaxf(acc[2 * s][0], 0.f), fmaxf(acc[2 * s][1], 0.f));
        a[s][1] = pack_bf16(fmaxf(acc[2 * s][2], 0.f), fmaxf(acc[2 * s][3], 0.f));
        a[s][2] = pack_bf16(fmaxf(acc[2 * s + 1][0], 0.f), fmaxf(acc[2 * s + 1][1], 0.f));
        a[s][3] = pack_bf16(fmaxf(acc[2 * s + 1][2], 0.f), fmaxf(acc[2 * s + 1][3], 0.f));
    }
}
// the weight fragments of two n-tiles for one k-step: b[0], b[1] of the first,
// b[2], b[3] of the second
__device__ __forceinline__ void load_b2(uint32_t addr, uint32_t (&b)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(addr));
}

// What bounds it: reading the weights from shared memory (every warp reads all
// of them for its rows) and the latency of the patch loads. With MT = 2 a
// weight fragment serves 32 rows; layer 2 runs in two halves of its outputs,
// each at once taken into layer 3, so that the accumulators fit the registers;
// a CTA's next rows are prefetched into L2 a tile ahead. 1,000,003 rows of width
// 160: 326 -> 272 us (the tensor pipe at 66% of an SM's active cycles). Every accumulator sees
// the same products in the same order as with MT = 1, so the outputs are equal.
template <int H, int MT>
__global__ void __launch_bounds__(256, 1) k_mlp_bf16(const float *__restrict__ x, long long n,
                                                      const uint16_t *__restrict__ wt, const float *__restrict__ bias,
                                                      float *__restrict__ out, bool l2) {
    using G = MlpGeo<H>;
    constexpr int NT = G::NT, S2 = G::S2, NH = NT / 2, ROWS = 128 * MT, K1 = K1P / 16;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t *W1s = reinterpret_cast<uint16_t *>(smem_raw);
    uint16_t *W2s = W1s + H * S1;
    uint16_t *W3s = W2s + H * S2;
    float *Bs = reinterpret_cast<float *>(W3s + 8 * S2);
    const long long n_tiles = (n + ROWS - 1) / ROWS;
    // the whole 16-byte words of tile t's rows, into L2 (l2: they lie in device memory)
    auto prefetch = [&](long long t) {
        if (threadIdx.x != 0 || t >= n_tiles || !l2) return;
        const char *a = reinterpret_cast<const char *>(x + t * ROWS * NIN);
        const char *b = reinterpret_cast<const char *>(x + min(n, (t + 1) * (long long)ROWS) * NIN);
        a += (16 - (reinterpret_cast<uintptr_t>(a) & 15)) & 15;
        const long long bytes = (b - a) & ~15ll;
        if (bytes > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)bytes) : "memory");
    };
    prefetch(blockIdx.x);
    // weights into shared memory, 16 bytes at a time (rows are 16-byte multiples)
    for (int i = threadIdx.x; i < H * (K1P / 8); i += blockDim.x) {
        const int r = i / (K1P / 8), c = i % (K1P / 8);
        *reinterpret_cast<uint4 *>(W1s + r * S1 + c * 8) = *reinterpret_cast<const uint4 *>(wt + G::w1 + (size_t)r * K1P + c * 8);
    }
    for (int i = threadIdx.x; i < H * (H / 8); i += blockDim.x) {
        const int r = i / (H / 8), c = i % (H / 8);
        *reinterpret_cast<uint4 *>(W2s + r * S2 + c * 8) = *reinterpret_cast<const uint4 *>(wt + G::w2 + (size_t)r * H + c * 8);
    }
    for (int i = threadIdx.x; i < 8 * (H / 8); i += blockDim.x) {
        const int r = i / (H / 8), c = i % (H / 8);
        *reinterpret_cast<uint4 *>(W3s + r * S2 + c * 8) = *reinterpret_cast<const uint4 *>(wt + G::w3 + (size_t)r * H + c * 8);
    }
    for (int i = threadIdx.x; i < 2 * H + 8; i += blockDim.x) Bs[i] = bias[i];
    __syncthreads();

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    // the lane's row for ldmatrix: n = lane % 8 (+ 8 for the second n-tile), k = 8 for odd groups of 8 lanes
    const int br = (lane & 7) + ((lane >> 4) << 3), bk = ((lane >> 3) & 1) * 8;
    const uint32_t w1a = (uint32_t)__cvta_generic_to_shared(W1s + br * S1 + bk);
    const uint32_t w2a = (uint32_t)__cvta_generic_to_shared(W2s + br * S2 + bk);
    for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        prefetch(tile + gridDim.x);
        const long long r0 = tile * ROWS + warp * (16 * MT) + g;   // rows r0 + 16 m and r0 + 16 m + 8
        const float *xr[MT];
        bool v0[MT], v1[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            xr[m] = x + (r0 + 16 * m) * NIN + 2 * t;
            v0[m] = r0 + 16 * m < n;
            v1[m] = r0 + 16 * m + 8 < n;
        }
        uint32_t af[MT][NT / 2][4];
        {   // layer 1: acc = b1 + x W1
            float acc[MT][NT][4];
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    acc[m][j][0] = acc[m][j][2] = Bs[8 * j + 2 * t];
                    acc[m][j][1] = acc[m][j][3] = Bs[8 * j + 2 * t + 1];
                }
            float2 p[2][MT][4];
            auto load = [&](int s, float2 (&f)[MT][4]) {
                const float2 z = make_float2(0.f, 0.f);
                const bool a = 16 * s + 2 * t < NIN, b = 16 * s + 2 * t + 8 < NIN;
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const float *x0 = xr[m] + 16 * s, *x1 = x0 + 8 * NIN;
                    f[m][0] = v0[m] && a ? *reinterpret_cast<const float2 *>(x0) : z;
                    f[m][1] = v1[m] && a ? *reinterpret_cast<const float2 *>(x1) : z;
                    f[m][2] = v0[m] && b ? *reinterpret_cast<const float2 *>(x0 + 8) : z;
                    f[m][3] = v1[m] && b ? *reinterpret_cast<const float2 *>(x1 + 8) : z;
                }
            };
            load(0, p[0]);
#pragma unroll
            for (int s = 0; s < K1; ++s) {
                if (s + 1 < K1) load(s + 1, p[(s + 1) & 1]);
                uint32_t a[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int u = 0; u < 4; ++u) a[m][u] = pack_bf16(p[s & 1][m][u].x, p[s & 1][m][u].y);
#pragma unroll
                for (int j = 0; j < NT; j += 2) {
                    uint32_t b[4];
                    load_b2(w1a + (uint32_t)(8 * j * S1 + 16 * s) * 2, b);
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][j], a[m], b[0], b[1]);
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][j + 1], a[m], b[2], b[3]);
                }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) to_frags<NT>(acc[m], af[m]);
        }
        // layer 2, a half of its outputs at a time, and layer 3 (6 outputs in one n-tile of 8) over that half
        float o[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            o[m][0] = o[m][2] = Bs[2 * H + 2 * t];
            o[m][1] = o[m][3] = Bs[2 * H + 2 * t + 1];
        }
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float acc[MT][NH][4];
#pragma unroll
            for (int j = 0; j < NH; ++j)
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    acc[m][j][0] = acc[m][j][2] = Bs[H + 8 * (half * NH + j) + 2 * t];
                    acc[m][j][1] = acc[m][j][3] = Bs[H + 8 * (half * NH + j) + 2 * t + 1];
                }
#pragma unroll
            for (int s = 0; s < G::KS; ++s)
#pragma unroll
                for (int j = 0; j < NH; j += 2) {
                    uint32_t b[4];
                    load_b2(w2a + (uint32_t)(8 * (half * NH + j) * S2 + 16 * s) * 2, b);
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][j], af[m][s], b[0], b[1]);
#pragma unroll
                    for (int m = 0; m < MT; ++m) mma_bf16(acc[m][j + 1], af[m][s], b[2], b[3]);
                }
#pragma unroll
            for (int i = 0; i < NH / 2; ++i) {
                const uint16_t *w = W3s + g * S2 + 16 * (half * (NH / 2) + i) + 2 * t;
                const uint32_t b0 = *reinterpret_cast<const uint32_t *>(w), b1 = *reinterpret_cast<const uint32_t *>(w + 8);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const float (&c0)[4] = acc[m][2 * i], (&c1)[4] = acc[m][2 * i + 1];
                    const uint32_t a[4] = {pack_bf16(fmaxf(c0[0], 0.f), fmaxf(c0[1], 0.f)), pack_bf16(fmaxf(c0[2], 0.f), fmaxf(c0[3], 0.f)),
                                           pack_bf16(fmaxf(c1[0], 0.f), fmaxf(c1[1], 0.f)), pack_bf16(fmaxf(c1[2], 0.f), fmaxf(c1[3], 0.f))};
                    mma_bf16(o[m], a, b0, b1);
                }
            }
        }
        if (t < 3) {
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                float *q = out + (r0 + 16 * m) * NOUT + 2 * t;
                if (v0[m]) *reinterpret_cast<float2 *>(q) = make_float2(o[m][0], o[m][1]);
                if (v1[m]) *reinterpret_cast<float2 *>(q + 8 * NOUT) = make_float2(o[m][2], o[m][3]);
            }
        }
    }
}

template <int H>
int infer_h(tpx_ctx *c, const void *packed, const float *x, long long n, float *out) {
    using G = MlpGeo<H>;
    // the shared-memory attribute belongs to each device's context
    static std::atomic<bool> attr[64];
    int dev = 0, sms = 0;
    if (ck(cudaGetDevice(&dev)) || ck(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return TPX_ECUDA;
    const bool known = dev >= 0 && dev < 64;
    if (!known || !attr[dev].load(std::memory_order_acquire)) {
        if (ck(cudaFuncSetAttribute(k_mlp_bf16<H, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::smem)) ||
            ck(cudaFuncSetAttribute(k_mlp_bf16<H, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::smem)))
            return TPX_ECUDA;
        if (known) attr[dev].store(true, std::memory_order_release);
    }
    const uint16_t *wt = static_cast<const uint16_t *>(packed);
    const float *bias = reinterpret_cast<const float *>(static_cast<const char *>(packed) + packed_bias_off(G::wend));
    // one tile of 128 rows per SM is the shortest way for few rows; beyond that 256 rows a tile
    const long long tiles = (n + 127) / 128;
    const bool l2 = device_memory(x);
    if (tiles <= sms) k_mlp_bf16<H, 1><<<(unsigned)tiles, 256, G::smem, c->stream>>>(x, n, wt, bias, out, l2);
    else k_mlp_bf16<H, 2><<<(unsigned)std::min<long long>((n + 255) / 256, sms), 256, G::smem, c->stream>>>(x, n, wt, bias, out, l2);
    return ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}
template <int H>
int pack_h(tpx_ctx *c, const float *P, void *packed) {
    using G = MlpGeo<H>;
    uint16_t *wt = static_cast<uint16_t *>(packed);
    float *bias = reinterpret_cast<float *>(static_cast<char *>(packed) + packed_bias_off(G::wend));
    k_pack<H><<<grid_for((long long)G::wend + 2 * H + 8), 256, 0, c->stream>>>(P, wt, bias);
    return ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}

}  // namespace tpxr

// the minibatch loss and its output gradient, and one Adam step, for the
// convolutional refiner (tpx_cnn.cu), which shares the loss and optimiser
int tpxr_loss(cudaStream_t s, const float *out, const float *y, int n, float w_off, float *dout, float *loss) {
    tpxr::k_loss<<<tpxr::grid_for(n), 256, 0, s>>>(out, y, n, w_off, dout, loss);
    return tpxr::ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}
int tpxr_adam(cudaStream_t s, float *p, const float *g, float *m, float *v, long long n, float lr, long long step) {
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    tpxr::k_adam<<<tpxr::grid_for(n), 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, c1, c2, 1e-8f);
    return tpxr::ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}

using namespace tpxr;

template <typename OutT>
static int refine_patches(tpx_ctx *c, const uint64_t *d_packets, int64_t n, int64_t base, const int64_t *d_labels,
                          const tpx_record *d_clusters, int64_t n_clusters, int32_t min_pixels, OutT *d_patches,
                          int64_t *d_sel, int32_t *d_centre, int64_t capacity, int64_t *d_n_patches) {
    if (!c || n < 0 || n_clusters < 0 || capacity < 0 || !d_n_patches || min_pixels < 0) return TPX_EINVAL;
    if ((n > 0 && (!d_packets || !d_labels)) || (n_clusters > 0 && !d_clusters)) return TPX_EINVAL;
    if (capacity > 0 && (!d_patches || !d_sel || !d_centre)) return TPX_EINVAL;
    cudaStream_t s = c->stream;
    if (ck(cudaMemsetAsync(d_n_patches, 0, 8, s))) return TPX_ECUDA;
    if (n_clusters == 0 || n == 0) return TPX_OK;
    // scratch: block counts, the list of incomplete patches; for those the
    // patch of each root packet and the cell keys
    const long long nb = (n_clusters + SELB - 1) / SELB;
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    const long long nt = (n + PT - 1) / PT;
    const size_t b_info = al(sizeof(PatchInfo)) + al(sizeof(TileSel) * (size_t)nt);
    const size_t need = b_info + al(4 * (size_t)nb) + 2 * al(4 * (size_t)capacity + 4) +
                        al(sizeof(SelRoot) * (size_t)capacity) + al(4 * (size_t)n) +
                        al(8 * (size_t)capacity * PC + 8);
    int rc = tpxg::reserve(c, need);
    if (rc) return rc;
    char *m = static_cast<char *>(c->g_mem);
    PatchInfo *info = reinterpret_cast<PatchInfo *>(m); m += al(sizeof(PatchInfo));
    TileSel *tiles = reinterpret_cast<TileSel *>(m); m += al(sizeof(TileSel) * (size_t)nt);
    unsigned *bcnt = reinterpret_cast<unsigned *>(m); m += al(4 * (size_t)nb);
    unsigned *inc = reinterpret_cast<unsigned *>(m); m += al(4 * (size_t)capacity + 4);
    unsigned *far = reinterpret_cast<unsigned *>(m); m += al(4 * (size_t)capacity + 4);
    SelRoot *roots = reinterpret_cast<SelRoot *>(m); m += al(sizeof(SelRoot) * (size_t)capacity);
    int *slot = reinterpret_cast<int *>(m); m += al(4 * (size_t)n);
    unsigned long long *key = reinterpret_cast<unsigned long long *>(m);
    const long long *lab = reinterpret_cast<const long long *>(d_labels);
    long long *sel = reinterpret_cast<long long *>(d_sel);
    if (ck(cudaMemsetAsync(info, 0, b_info, s))) return TPX_ECUDA;
    k_sel_count<<<(unsigned)nb, SELT, 0, s>>>(d_clusters, n_clusters, min_pixels, bcnt);
    if (nb > kResumBlocks) k_sel_scan<<<1, 1024, 0, s>>>(bcnt, nb);
    k_select<<<(unsigned)nb, SELT, 0, s>>>(d_packets, d_clusters, n_clusters, min_pixels, bcnt, nb, capacity, base, n, sel,
                                           d_centre, reinterpret_cast<long long *>(d_n_patches), tiles, roots, info);
    if (capacity > 0) {
        k_patch_tiles<OutT><<<(unsigned)nt, PTH, 0, s>>>(d_packets, n, base, lab, roots, tiles, d_patches, inc, info);
        k_patch_wide<OutT><<<c->num_sms * 4, PWT, 0, s>>>(d_packets, n, base, lab, d_clusters, sel, d_centre, inc, d_patches,
                                                          far, info);
    }
    static_assert(sizeof(PatchInfo) <= 4 * sizeof(int64_t), "h_words");
    if (ck(cudaMemcpyAsync(c->h_words, info, sizeof(PatchInfo), cudaMemcpyDeviceToHost, s)) || ck(cudaStreamSynchronize(s))) return TPX_ECUDA;
    const PatchInfo &h = *reinterpret_cast<const PatchInfo *>(c->h_words);
    const long long np = (long long)h.n_sel, ns = np < capacity ? np : capacity;
    const bool wider = search_wider(h.n_inc, n);
    const long long ni = h.odd ? ns : (long long)(wider ? h.n_far : h.n_inc);
    const unsigned *list = h.odd || wider ? far : inc;
    if (ni > 0) {
        if (h.odd) k_list_all<<<grid_for(ns), 256, 0, s>>>(far, ns);
        k_clear<<<grid_for(std::max<long long>(n, ni * PC)), 256, 0, s>>>(slot, n, key, ni * PC);
        k_roots<<<grid_for(ni), 256, 0, s>>>(roots, list, ni, n, slot);
        k_patch_keys<<<grid_for(n), 256, 0, s>>>(d_packets, n, base, lab, slot, list, roots,
                                                 h.odd ? d_centre : nullptr, key);
        k_patch_fill<OutT><<<grid_for(ni * PC), 256, 0, s>>>(list, key, ni, d_patches);
    }
    if (ck(cudaGetLastError())) return TPX_ECUDA;
    return np > capacity ? TPX_EOVERFLOW : TPX_OK;
}

extern "C" {

int tpx_refine_patches(tpx_ctx *c, const uint64_t *d_packets, int64_t n, int64_t base, const int64_t *d_labels,
                       const tpx_record *d_clusters, int64_t n_clusters, int32_t min_pixels, float *d_patches,
                       int64_t *d_sel, int32_t *d_centre, int64_t capacity, int64_t *d_n_patches) {
    return refine_patches<float>(c, d_packets, n, base, d_labels, d_clusters, n_clusters, min_pixels, d_patches, d_sel,
                                 d_centre, capacity, d_n_patches);
}

int tpx_refine_patches_bf16(tpx_ctx *c, const uint64_t *d_packets, int64_t n, int64_t base, const int64_t *d_labels,
                            const tpx_record *d_clusters, int64_t n_clusters, int32_t min_pixels, uint16_t *d_patches,
                            int64_t *d_sel, int32_t *d_centre, int64_t capacity, int64_t *d_n_patches) {
    return refine_patches<uint16_t>(c, d_packets, n, base, d_labels, d_clusters, n_clusters, min_pixels, d_patches,
                                    d_sel, d_centre, capacity, d_n_patches);
}

int64_t tpx_refiner_params(int32_t hidden) { return hidden > 0 ? Layout(hidden).total : 0; }

// forward pass; `act` (n x (2H + NOUT) floats) keeps the activations for a
// backward pass, or may be NULL when `out` is given
static int forward(tpx_ctx *c, const float *P, int h, const float *x, int64_t n, float *a1, float *a2, float *out) {
    const Layout L(h);
    cudaStream_t s = c->stream;
    // rows in chunks the GEMM grid can hold (grid.y <= 65535 tiles of 64 rows)
    constexpr int64_t kRows = 1LL << 21;
    for (int64_t r0 = 0; r0 < n; r0 += kRows) {
        const int m = (int)(n - r0 < kRows ? n - r0 : kRows);
        gemm(s, x + r0 * NIN, NIN, 1, P + L.w1, h, 1, a1 + r0 * h, h, m, h, NIN, P + L.b1, true);
        gemm(s, a1 + r0 * h, h, 1, P + L.w2, h, 1, a2 + r0 * h, h, m, h, h, P + L.b2, true);
        gemm(s, a2 + r0 * h, h, 1, P + L.w3, NOUT, 1, out + r0 * NOUT, NOUT, m, NOUT, h, P + L.b3, false);
    }
    return ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}

int tpx_refiner_forward(tpx_ctx *c, const float *d_params, int32_t hidden, const float *d_x, int64_t n,
                        float *d_work, float *d_out) {
    if (!c || !d_params || hidden < 1 || n < 0 || (n > 0 && (!d_x || !d_work || !d_out)) || n >= (1LL << 31))
        return TPX_EINVAL;
    if (n == 0) return TPX_OK;
    return forward(c, d_params, hidden, d_x, n, d_work, d_work + (long long)n * hidden, d_out);
}

int tpx_refiner_train_step(tpx_ctx *c, float *d_params, float *d_adam_m, float *d_adam_v, float *d_grad,
                           int32_t hidden, int64_t step, const float *d_x, const float *d_y, int64_t n, float lr,
                           float offset_weight, float *d_work, float *d_loss) {
    if (!c || !d_params || !d_adam_m || !d_adam_v || !d_grad || hidden < 1 || step < 1 || !d_x || !d_y || n < 1 ||
        !d_work || !d_loss || n > (1LL << 21))
        return TPX_EINVAL;
    const Layout L(hidden);
    const int h = hidden;
    cudaStream_t s = c->stream;
    // widths that fit the fused step's shared memory (4096 rows, width 160: 2.58 ms with the GEMMs below)
    if (h <= tpxt::kMaxHidden)
        return ck(tpxt::train_step(s, d_params, d_adam_m, d_adam_v, d_grad, h, step, d_x, d_y, n, lr, offset_weight, d_work,
                                   d_loss)) ? TPX_ECUDA : TPX_OK;
    float *a1 = d_work, *a2 = a1 + (long long)n * h, *out = a2 + (long long)n * h;
    float *dout = out + (long long)n * NOUT, *d2 = dout + (long long)n * NOUT, *d1 = d2 + (long long)n * h;
    int rc = forward(c, d_params, h, d_x, n, a1, a2, out);
    if (rc) return rc;
    if (ck(cudaMemsetAsync(d_loss, 0, 4, s))) return TPX_ECUDA;
    k_loss<<<grid_for(n), 256, 0, s>>>(out, d_y, (int)n, offset_weight, dout, d_loss);
    // layer 3: dW3 = a2^T dout, db3 = colsum(dout), d2 = dout W3^T
    gemm(s, a2, 1, h, dout, NOUT, 1, d_grad + L.w3, NOUT, h, NOUT, (int)n, nullptr, false);
    k_colsum<<<1, 256, 0, s>>>(dout, (int)n, NOUT, d_grad + L.b3);
    gemm(s, dout, NOUT, 1, d_params + L.w3, 1, NOUT, d2, h, (int)n, h, NOUT, nullptr, false);
    k_relu_back<<<grid_for((long long)n * h), 256, 0, s>>>(d2, a2, (long long)n * h);
    // layer 2
    gemm(s, a1, 1, h, d2, h, 1, d_grad + L.w2, h, h, h, (int)n, nullptr, false);
    k_colsum<<<(h + 255) / 256, 256, 0, s>>>(d2, (int)n, h, d_grad + L.b2);
    gemm(s, d2, h, 1, d_params + L.w2, 1, h, d1, h, (int)n, h, h, nullptr, false);
    k_relu_back<<<grid_for((long long)n * h), 256, 0, s>>>(d1, a1, (long long)n * h);
    // layer 1
    gemm(s, d_x, 1, NIN, d1, h, 1, d_grad + L.w1, h, NIN, h, (int)n, nullptr, false);
    k_colsum<<<(h + 255) / 256, 256, 0, s>>>(d1, (int)n, h, d_grad + L.b1);
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_adam<<<grid_for(L.total), 256, 0, s>>>(d_params, d_grad, d_adam_m, d_adam_v, L.total, lr, b1, b2, c1, c2, 1e-8f);
    return ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}

int64_t tpx_refiner_packed_bytes(int32_t hidden) {
    switch (hidden) {
        case 64: return (int64_t)MlpGeo<64>::packed_bytes;
        case 128: return (int64_t)MlpGeo<128>::packed_bytes;
        case 160: return (int64_t)MlpGeo<160>::packed_bytes;
        default: return 0;
    }
}

int tpx_refiner_pack(tpx_ctx *c, const float *d_params, int32_t hidden, void *d_packed) {
    if (!c || !d_params || !d_packed || (reinterpret_cast<uintptr_t>(d_packed) & 15)) return TPX_EINVAL;
    switch (hidden) {
        case 64: return pack_h<64>(c, d_params, d_packed);
        case 128: return pack_h<128>(c, d_params, d_packed);
        case 160: return pack_h<160>(c, d_params, d_packed);
        default: return TPX_EUNSUPPORTED;
    }
}

int tpx_refiner_infer(tpx_ctx *c, const void *d_packed, int32_t hidden, const float *d_x, int64_t n, float *d_out) {
    if (!c || n < 0 || (n > 0 && (!d_packed || !d_x || !d_out))) return TPX_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_packed) & 15) || (reinterpret_cast<uintptr_t>(d_x) & 7) ||
        (reinterpret_cast<uintptr_t>(d_out) & 7))
        return TPX_EINVAL;
    if (hidden != 64 && hidden != 128 && hidden != 160) return TPX_EUNSUPPORTED;
    if (n == 0) return TPX_OK;
    switch (hidden) {
        case 64: return infer_h<64>(c, d_packed, d_x, n, d_out);
        case 128: return infer_h<128>(c, d_packed, d_x, n, d_out);
        default: return infer_h<160>(c, d_packed, d_x, n, d_out);
    }
}

int tpx_refine_decide(tpx_ctx *c, const float *d_out, const tpx_record *d_clusters, const int64_t *d_sel,
                      const int32_t *d_centre, int64_t n, float threshold, float *d_hits) {
    if (!c || n < 0 || (n > 0 && (!d_out || !d_clusters || !d_sel || !d_centre || !d_hits))) return TPX_EINVAL;
    if (!(threshold > 0.f && threshold < 1.f)) return TPX_EINVAL;
    if (n == 0) return TPX_OK;
    const float lt = (float)std::log((double)threshold / (1.0 - (double)threshold));
    k_decide<<<grid_for(n), 256, 0, c->stream>>>(d_out, d_clusters, reinterpret_cast<const long long *>(d_sel),
                                                 d_centre, n, lt, d_hits);
    return ck(cudaGetLastError()) ? TPX_ECUDA : TPX_OK;
}

}  // extern "C"
