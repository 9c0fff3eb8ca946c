// CUDA kernels of the improved W-stacking hot path (sm_103a).
//
// Gridding (Algorithm 5):   prep and count -> sort -> per plane chunk: grid3d -> inv_cols -> inv_rows
//                           (transforms.cu: inverse DFTs, crop, x exp(2 pi i t z), sum over t,
//                           x h_x h_y h_z)
// Degridding (Algorithm 6): prep and count -> sort -> per plane chunk: fwd_rows -> fwd_cols
//                           (transforms.cu: x h_x h_y h_z, x exp(-2 pi i t z), zero pad, forward DFTs)
//                           -> degrid3d (3-D correlation with C_x C_y C_z, x exp(-2 pi i w (n0-1)))
//
// Grid indices: row s (v direction) and column r (u direction) of a plane are
// stored modulo N'.  Because exp(2 pi i r j / N') is N'-periodic in r, a tap
// that runs past the grid edge wraps onto the opposite edge and the inverse
// DFT of the wrapped grid is exactly the sum over all integers r of Eq.
// gridded-dirty-map; the centred crop |x| < x0 is then rows/columns
// [N'-N/2, N') and [0, N/2).  Planes use the column-block layout of common.cuh.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "ws_internal.hpp"

namespace ws {
namespace {

// An integer-valued double (|x| < 1e15) modulo n in [0, n): integer arithmetic,
// with the division only for the rare points more than a grid away.
__device__ __forceinline__ int wrap_index(double x, int n) {
    long long i = (long long)x;
    if (i < -n || i >= 2LL * n) i %= n;
    if (i < 0) i += n;
    if (i >= n) i -= n;
    return (int)i;
}

// ---------------------------------------------------------------------------
// Binning: counting sort of (visibility, bin) pairs by bin id
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t tile_id(const Launch &L, int tt, int tv, int tu) {
    return ((uint32_t)tt * L.ntv + tv) * L.ntu + tu;
}

// Gridding bin: a tile column (tv, tu) and the t-tile of the first tap.  A
// column's bins are contiguous, in t order.
__device__ __forceinline__ uint32_t column_bin(const Launch &L, int tv, int tu, int tt) {
    return ((uint32_t)tv * L.ntu + tu) * L.ntt + tt;
}

// The tile columns a footprint's W x W taps in (u, v) touch: 1 or 2 along each axis.
__device__ __forceinline__ void footprint_columns(const Launch &L, const VisRec &r, int *tu, int &nu_, int *tv,
                                                  int &nv_) {
    tu[0] = r.r0 / TU;
    tu[1] = wrap_add(r.r0, L.W - 1, L.Np) / TU;
    nu_ = tu[1] != tu[0] ? 2 : 1;
    tv[0] = r.s0 >> L.tv_log;
    tv[1] = wrap_add(r.s0, L.W - 1, L.Np) >> L.tv_log;
    nv_ = tv[1] != tv[0] ? 2 : 1;
}

// Bins of a record: its tile columns with the first tap's t-tile (grid), or
// the tile of its first tap (degrid).
template <bool GRID>
__device__ __forceinline__ int record_keys(const Launch &L, const VisRec &r, uint32_t *keys) {
    if (r.t0 < 0) return 0;
    if (!GRID) {
        keys[0] = tile_id(L, r.t0 / TT, r.s0 >> L.tv_log, r.r0 / TU);
        return 1;
    }
    int tu[2], tv[2], nu_, nv_;
    footprint_columns(L, r, tu, nu_, tv, nv_);
    int n = 0;
    for (int b = 0; b < nv_; ++b)
        for (int a = 0; a < nu_; ++a) keys[n++] = column_bin(L, tv[b], tu[a], r.t0 / TT);
    return n;
}

constexpr int kMaxKeys = 2 * 2;

// Counts the record's bins and marks the stack tiles its footprint touches.
// Every other cell of the stack is zero when gridding and never read when
// degridding, so the plane kernels skip it.
template <bool GRID>
__device__ __forceinline__ void count_record(const Launch &L, const VisRec &r, uint32_t *__restrict__ counts,
                                             uint8_t *__restrict__ tile_occ) {
    uint32_t keys[kMaxKeys];
    const int n = record_keys<GRID>(L, r, keys);
    for (int i = 0; i < n; ++i) atomicAdd(&counts[keys[i]], 1u);
    if (n == 0) return;
    int tu[2], tv[2], nu_, nv_;
    footprint_columns(L, r, tu, nu_, tv, nv_);
    const int tt1 = (r.t0 + L.W - 1) / TT;
    for (int tt = r.t0 / TT; tt <= tt1; ++tt)
        for (int b = 0; b < nv_; ++b)
            for (int a = 0; a < nu_; ++a) tile_occ[tile_id(L, tt, tv[b], tu[a])] = 1;   // stores only: no waits
}

// ---------------------------------------------------------------------------
// Pre-processing (Section 3.3 tap rule, Section 5.2 scaling and pre-phase)
// ---------------------------------------------------------------------------
// What prep_kernel makes of a record once it has it: nothing more (the bound
// set's records), or its degridding or gridding bins counted and its tiles marked.
enum : int { kPrepOnly = 0, kPrepDegrid = 1, kPrepGrid = 2 };

// The tap rule's floor(x + W/2) for |x| < 2^51 and, in nu, the offset x + (W-1)/2 -
// floor(x + W/2) in [-1/2, 1/2), from FP64 adds alone: the nearest integer to x +
// (W-1)/2 comes from adding 1.5 x 2^52 (it is left in the sum's low bits), and
// differs from the floor only where x + W/2 is an integer and the tie went down.
// FP64 arithmetic is what bounds the kernel (GB300 does 0.6 T FP64 operations a
// second), floor and the conversions to integers more so.
__device__ __forceinline__ void tap_floor(double x, double half_wm1, int *floor_low, float *nu) {
    constexpr double kRound = 6755399441055744.0;
    const double y = x + half_wm1, s = y + kRound;
    double d = y - (s - kRound);
    int low = __double2loint(s);
    if (d == 0.5) {
        d = -0.5;
        ++low;
    }
    *floor_low = low;
    *nu = (float)d;
}

// |x| below about 10^9 (an exponent below 30), by integer comparison: false for NaN and infinities too.
__device__ __forceinline__ bool small_enough(double x) {
    return (__double2hiint(x) & 0x7fffffff) < ((1023 + 30) << 20);
}

// A grid index i (|i| < 2^31) modulo n: with the division only for the rare points more than a grid away.
__device__ __forceinline__ int wrap_small(int i, int n) {
    if (i < -n || i >= 2 * n) i %= n;
    if (i < 0) i += n;
    return i >= n ? i - n : i;
}

// The loop bound: M records, 8 CTAs per SM in a grid-stride loop, so that the
// plan's constants in FP64 (W / 2, offsets) are formed once per thread, not once
// per visibility.  FP64 arithmetic is what bounds this kernel (GB300 adds and
// multiplies 0.6 T FP64 numbers a second).
template <int BIN>
__global__ void prep_kernel(Launch L, const double *__restrict__ uvw, const float2 *__restrict__ vis,
                            int64_t M, VisRec *__restrict__ rec, unsigned long long *__restrict__ drop,
                            uint32_t *__restrict__ counts, uint8_t *__restrict__ tile_occ, float2 *__restrict__ zeroed) {
    const int W = L.W;
    const double half_w = 0.5 * W, half_wm1 = 0.5 * (W - 1);
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < M; k += (int64_t)gridDim.x * blockDim.x) {
        double u = uvw[3 * k], v = uvw[3 * k + 1], w = uvw[3 * k + 2];
        if (BIN == kPrepDegrid) zeroed[k] = make_float2(0.f, 0.f);      // the output that degridding adds to
        // Section 5.4, real sky: V(u, v, w) = conj V(-u, -v, -w), so w < 0 is gridded at
        // -(u, v, w) with the conjugate value (and degridded there, conjugated afterwards)
        const bool folded = L.fold && w < 0.0;
        if (folded) {
            u = -u;
            v = -v;
            w = -w;
        }
        VisRec r;
        r.r0 = r.s0 = 0;
        r.t0 = -1;
        r.nux = r.nuy = r.nuz = 0.f;
        r.vre = r.vim = 0.f;
        const double up = u * L.uv_scale, vp = v * L.uv_scale, wp = w * L.nscale;
        const bool near = small_enough(up) && small_enough(vp);
        if (!near && (!(fabs(up) < 1e15) || !(fabs(vp) < 1e15))) {   // also catches NaN
            atomicAdd(&drop[0], 1ull);
            rec[k] = r;
            continue;
        }
        int it;
        float nuz;
        tap_floor(wp, half_wm1, &it, &nuz);
        const int t0 = it - (W - 1) - L.t_lo;
        if (!small_enough(wp) || t0 < 0 || t0 > L.Nw - W) {          // NaN w is not small
            atomicAdd(&drop[1], 1ull);
            rec[k] = r;
            continue;
        }
        r.t0 = t0;
        r.nuz = nuz;
        if (near) {
            int iu, iv;
            tap_floor(up, half_wm1, &iu, &r.nux);
            tap_floor(vp, half_wm1, &iv, &r.nuy);
            r.r0 = wrap_small(iu - (W - 1), L.Np);
            r.s0 = wrap_small(iv - (W - 1), L.Np);
        } else {
            const double fu = floor(up + half_w), fv = floor(vp + half_w);
            r.r0 = wrap_index(fu - (W - 1), L.Np);
            r.s0 = wrap_index(fv - (W - 1), L.Np);
            r.nux = (float)(up + half_wm1 - fu);
            r.nuy = (float)(vp + half_wm1 - fv);
        }
        // pre-phase exp(+2 pi i w (n0 - 1)), argument reduced in FP64
        double turns = w * L.n0m1;
        turns -= (turns + 6755399441055744.0) - 6755399441055744.0;      // |turns| < 2^51: rint by 1.5 x 2^52
        float s, c;
        sincospif(2.0f * (float)turns, &s, &c);
        if (BIN == kPrepGrid) {
            float2 V = vis[k];
            if (folded) V.y = -V.y;
            r.vre = V.x * c - V.y * s;
            r.vim = V.x * s + V.y * c;
        } else {
            r.vre = c;          // conjugate phase applied after degridding
            r.vim = -s;
        }
        rec[k] = r;
        if (BIN == kPrepGrid) count_record<true>(L, r, counts, tile_occ);
        if (BIN == kPrepDegrid) count_record<false>(L, r, counts, tile_occ);
    }
}

// Zeroes the counts and the occupancy maps, and the drop counters if there are any.
__global__ void clear_bins_kernel(uint32_t *__restrict__ counts, int64_t n, uint8_t *__restrict__ tile_occ, int64_t nt,
                                  uint8_t *__restrict__ col_occ, int64_t nc, unsigned long long *__restrict__ drop) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < n; i += step) counts[i] = 0u;
    for (int64_t i = i0; i < nt / 16; i += step) reinterpret_cast<uint4 *>(tile_occ)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = nt / 16 * 16 + i0; i < nt; i += step) tile_occ[i] = 0;
    for (int64_t i = i0; i < nc; i += step) col_occ[i] = 0;
    if (drop && i0 < kCounters) drop[i0] = 0ull;
}

// The counting pass over records that are there already (the bound set's).
template <bool GRID>
__global__ void count_kernel(Launch L, const VisRec *__restrict__ rec, int64_t M, uint32_t *__restrict__ counts,
                             uint8_t *__restrict__ tile_occ) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < M) count_record<GRID>(L, rec[k], counts, tile_occ);
}

// Gridding records of a bound visibility set: the set's records hold the
// degridding factor exp(-2 pi i w (n0 - 1)); gridding needs V exp(+2 pi i w
// (n0 - 1)), with V conjugated where a real-sky plan folded w < 0.
__global__ void bound_grid_records_kernel(Launch L, const double *__restrict__ uvw, const float2 *__restrict__ vis,
                                          int64_t M, const VisRec *__restrict__ brec, VisRec *__restrict__ rec) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    VisRec r = brec[k];
    float2 V = vis[k];
    if (L.fold && uvw[3 * k + 2] < 0.0) V.y = -V.y;
    const float c = r.vre, s = -r.vim;      // exp(+2 pi i w (n0 - 1)) = (c, s)
    r.vre = V.x * c - V.y * s;
    r.vim = V.x * s + V.y * c;
    rec[k] = r;
}

// Lists the pairs: a bin's next place is its cursor, which starts at the bin's
// offset.  The CTAs from vis_blocks on mark the occupied (t-tile, u-tile) strips
// of N' rows (any tile of the strip touched) on the side.
template <bool GRID>
__global__ void scatter_kernel(Launch L, const VisRec *__restrict__ rec, int64_t M, int vis_blocks,
                               uint32_t *__restrict__ cursor, uint32_t *__restrict__ list,
                               const uint8_t *__restrict__ tile_occ, int64_t ntiles, uint8_t *__restrict__ col_occ) {
    if ((int)blockIdx.x >= vis_blocks) {
        const int64_t t = (int64_t)(blockIdx.x - vis_blocks) * blockDim.x + threadIdx.x;
        if (t >= ntiles || !tile_occ[t]) return;
        const int64_t c = (t / ((int64_t)L.ntu * L.ntv)) * L.ntu + t % L.ntu;
        if (!col_occ[c]) col_occ[c] = 1;
        return;
    }
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    uint32_t keys[kMaxKeys];
    int n = record_keys<GRID>(L, rec[k], keys);
    for (int i = 0; i < n; ++i) list[atomicAdd(&cursor[keys[i]], 1u)] = (uint32_t)k;
}

// Statistics only (WS_FLAG_TIMING): occupied tiles and occupied (t-tile,
// u-strip) strips of one t-tile per CTA.
__global__ void occ_count_kernel(Launch L, const uint8_t *__restrict__ tile_occ, const uint8_t *__restrict__ col_occ,
                                 uint32_t *__restrict__ counts) {
    const int tt = blockIdx.x;
    const int64_t per = (int64_t)L.ntu * L.ntv;
    uint32_t tiles = 0, strips = 0;
    for (int64_t i = threadIdx.x; i < per; i += blockDim.x) tiles += tile_occ[tt * per + i];
    for (int i = threadIdx.x; i < L.ntu; i += blockDim.x) strips += col_occ[(int64_t)tt * L.ntu + i];
    for (int o = 16; o > 0; o >>= 1) {
        tiles += __shfl_xor_sync(0xffffffffu, tiles, o);
        strips += __shfl_xor_sync(0xffffffffu, strips, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&counts[2 * tt], tiles);
        atomicAdd(&counts[2 * tt + 1], strips);
    }
}

// Exclusive scan of n uint32 (n <= 4096 * 4096): per-block scan of 4096
// elements, scan of the block sums in one block, then add back.
constexpr int kScanThreads = 1024;
constexpr int kScanPerBlock = 4 * kScanThreads;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total) {
    __shared__ uint32_t warp_sums[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = warp_sums[lane];
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    uint32_t before = (wid ? warp_sums[wid - 1] : 0u) + x - v;
    *total = warp_sums[31];
    __syncthreads();
    return before;
}

// (the counts are replaced by a copy of the offsets, the scatter's cursors)
__global__ void __launch_bounds__(kScanThreads) scan_block_kernel(uint32_t *__restrict__ counts,
                                                                  uint32_t *__restrict__ out,
                                                                  uint32_t *__restrict__ sums, int64_t n) {
    const int64_t base = (int64_t)blockIdx.x * kScanPerBlock + 4 * threadIdx.x;
    uint32_t a[4];
    for (int i = 0; i < 4; ++i) a[i] = base + i < n ? counts[base + i] : 0u;
    uint32_t local = a[0] + a[1] + a[2] + a[3], total;
    uint32_t run = block_exclusive_scan(local, &total);
    for (int i = 0; i < 4; ++i) {
        if (base + i < n) out[base + i] = counts[base + i] = run;
        run += a[i];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(uint32_t *sums, int nb) {
    const int base = 4 * threadIdx.x;
    uint32_t a[4];
    for (int i = 0; i < 4; ++i) a[i] = base + i < nb ? sums[base + i] : 0u;
    uint32_t total;
    uint32_t run = block_exclusive_scan(a[0] + a[1] + a[2] + a[3], &total);
    for (int i = 0; i < 4; ++i) {
        if (base + i < nb) sums[base + i] = run;
        run += a[i];
    }
}

__global__ void scan_add_kernel(uint32_t *__restrict__ out, uint32_t *__restrict__ cursor,
                                const uint32_t *__restrict__ sums, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = cursor[i] = out[i] + sums[i / kScanPerBlock];
}

// ---------------------------------------------------------------------------
// Gridding: Algorithm 5 steps 2 and 3a (Eq. gridded_vis).  One CTA owns one
// tile column -- TU grid columns x tv grid rows through every w-plane of the
// plane chunk -- and walks the column's bins in t order.  A bin holds the
// visibilities whose first tap lies in one t-tile, so their footprints reach
// at most TT + W - 1 consecutive planes: the CTA accumulates in a
// shared-memory ring of that many planes (plane t at ring slot t mod (TT + W
// - 1)), and before it adds a bin it writes out the planes that bin can no
// longer reach -- each occupied tile of the stack exactly once -- and clears
// their slots.  A visibility is one entry in each tile column its W x W taps
// in (u, v) touch (at most 2 x 2), whatever the planes its W taps in w span.
//
// A bin's entries are split evenly over the CTA's warps; a warp takes its
// share in chunks of up to kChunk entries, in three steps:
//   1. lane j prepares entry j of the chunk: its record, the part of its
//      W x W x W footprint that lies in the column and in the plane chunk
//      (first tap and tap count along u, v and w) and that part's first cell;
//   2. the warp evaluates the chunk's 3W weight polynomials C(r - u'),
//      C(s - v'), C(t - w'), one (entry, slot) pair per lane and round;
//   3. entry after entry, the lanes take the (row, plane) pairs of the part,
//      form C_y C_z V once each, and add C_x C_y C_z V along the part's run of
//      u taps with shared-memory reductions at immediate offsets.
// So the tap rule, the index arithmetic and the polynomials cost once per
// entry, and each tap costs one weight product and one reduction per
// component.
// ---------------------------------------------------------------------------
static_assert(kMaxDeg + 1 <= kCoefStride && kCoefStride % 4 == 0 && kMaxDeg == 16,
              "the Horner steps below read coefficients 0..16 as five float4");
static_assert(kMaxW <= 15, "tap counts and first taps are packed in 4 bits");
static_assert(ring_planes(kMaxW) <= 31, "ring slots are packed in 5 bits");
constexpr int kGeneral = -1;                       // item shape: the part wraps an axis of a small grid

// Dynamic shared memory of grid3d<W, R, DET> (grid_smem_bytes): the ring (re,
// im; FP32 sums, or the low and high words of 64-bit fixed-point sums for the deterministic mode), the
// weight table, and per warp the staged chunk (weights, items, values, nu).
template <int W, int R, bool DET>
struct GridSmem {
    static constexpr int S = 3 * W;                // weight slots per entry: u taps, v taps, w taps
    static constexpr int WX = wx_span(W);          // staged u weights, from the part's first tap
    static constexpr int SP = stage_stride(W);     // entry stride of the staged weights: u, v, w
    static constexpr int HI = ring_planes(W) * plane_stride(R) * 4;    // DET: from a sum's low word to its high word
    static constexpr int RP = ring_planes(W);      // ring planes
    static constexpr int PS = plane_stride(R);     // cells per ring plane (padded)
    static constexpr size_t re = 0;
    static constexpr size_t im = re + ring_bytes(W, R, DET);
    static constexpr size_t coef = im + ring_bytes(W, R, DET);
    static constexpr size_t wt = coef + (size_t)S * kCoefStride * 4;
    static constexpr size_t item = wt + (size_t)kGridWarps * kChunk * SP * 4;
    static constexpr size_t val = item + (size_t)kGridWarps * kChunk * 16;
    static constexpr size_t nu = val + (size_t)kGridWarps * kChunk * 8;
    static constexpr size_t bytes = nu + (size_t)kGridWarps * kChunk * 16;
    static_assert(bytes == grid_smem_bytes(W, R, DET), "the host's size of the gridding shared memory");
    static_assert(coef % 16 == 0 && wt % 16 == 0 && item % 16 == 0 && nu % 16 == 0, "float4 / int4 alignment");
};

// Taps [a0, a1) of a footprint that land in a tile, at tile-local index a - off.
struct Span {
    int a0, a1, off;
};

// The footprint covers positions first .. first + W - 1 and the tile org ..
// org + T - 1 of a periodic axis of length n >= T: the tile starts d = org -
// first (mod n) past the footprint's start, and if it runs past n it also
// covers the footprint's first d + T - n positions.  Returns 0, 1 or 2 spans
// (two only when n < W + T, a grid of 32 rows).
__device__ __forceinline__ int tile_spans(int org, int first, int n, int W, int T, Span &s0, Span &s1) {
    int d = org - first;
    if (d < 0) d += n;
    const Span inside{d, min(W, d + T), d}, wrapped{0, min(W, d + T - n), d - n};
    const bool has_inside = d < W, has_wrapped = d + T > n;
    s0 = has_inside ? inside : wrapped;
    s1 = wrapped;
    return (int)has_inside + (int)has_wrapped;
}

// Shared-memory FP32 add with no returned value, at a byte offset fixed at compile time.
template <int OFF>
__device__ __forceinline__ void red_shared_at(unsigned addr, float v) {
    asm volatile("red.shared.add.f32 [%0+%1], %2;" ::"r"(addr), "n"(OFF), "f"(v) : "memory");
}

// The 64-bit integer nearest v (ties to even), |v| < 2^62.  The conversion to 64 bits
// goes at the rate of FP64 arithmetic, and bounded the deterministic mode (120,960
// visibilities, W = 7, N = 512: 350 us with it, 274 so); this takes the two words of |v|
// by 32-bit conversions, both exact but for the low word's rounding (below 2^24 |v| is
// all in the low word; from there on it is an integer).
__device__ __forceinline__ long long nearest_int64(float v) {
    const float a = fabsf(v), x = a * 0x1p-32f;
    const unsigned hi = __float2uint_rz(x), lo = __float2uint_rn(fmaf(truncf(x), -0x1p32f, a));
    const long long q = (long long)((unsigned long long)hi << 32 | lo);
    return v < 0.f ? -q : q;
}
// The deterministic mode's shared-memory add: a contribution, in units of the
// column's 2^-scale, becomes the nearest 64-bit integer, and integer sums do not
// depend on the order of their terms.  A sum is kept as two 32-bit words `HI` bytes
// apart: shared memory adds 32-bit integers itself, while a 64-bit add is a loop of
// compare-and-swap.  Every addition to the low word adds its carry to the high
// word, so the pair is the 64-bit sum once all have arrived.
// add_low returns the low word before the addition; add_high takes it.
template <int OFF>
__device__ __forceinline__ unsigned add_low(unsigned addr, long long q) {
    unsigned old;
    asm volatile("atom.shared.add.u32 %0, [%1+%2], %3;" : "=r"(old) : "r"(addr), "n"(OFF), "r"((unsigned)q) : "memory");
    return old;
}
template <int OFF>
__device__ __forceinline__ void add_high(unsigned addr, long long q, unsigned old) {
    const unsigned carry = old + (unsigned)q < old ? 1u : 0u;
    asm volatile("red.shared.add.u32 [%0+%1], %2;" ::"r"(addr), "n"(OFF), "r"((unsigned)(q >> 32) + carry) : "memory");
}

// One contribution to a ring cell component at byte address addr (the general path: any v).
template <bool DET, int HI>
__device__ __forceinline__ void add_cell(unsigned addr, float v) {
    if constexpr (DET) {
        const long long q = __float2ll_rn(v);
        add_high<HI>(addr, q, add_low<0>(addr, q));
    } else {
        red_shared_at<0>(addr, v);
    }
}

// Adds p x wx[a] to cells a = 0 .. na - 1 of a ring row (byte address `addr`).
template <int W, int A = 0>
__device__ __forceinline__ void add_row(unsigned addr, const float (&wx)[wx_span(W)], int na, float p) {
    if constexpr (A < W) {
        if (A < na) {
            red_shared_at<4 * A>(addr, p * wx[A]);
            add_row<W, A + 1>(addr, wx, na, p);
        }
    }
}
// The same in fixed point: all low words first, so their returns are waited for once.
template <int W, int HI, int A = 0>
__device__ __forceinline__ void add_row_low(unsigned addr, const float (&wx)[wx_span(W)], int na, float p,
                                            long long (&q)[W], unsigned (&old)[W]) {
    if constexpr (A < W) {
        if (A < na) {
            q[A] = nearest_int64(p * wx[A]);
            old[A] = add_low<4 * A>(addr, q[A]);
            add_row_low<W, HI, A + 1>(addr, wx, na, p, q, old);
        }
    }
}
template <int W, int HI, int A = 0>
__device__ __forceinline__ void add_row_high(unsigned addr, int na, const long long (&q)[W], const unsigned (&old)[W]) {
    if constexpr (A < W) {
        if (A < na) {
            add_high<HI + 4 * A>(addr, q[A], old[A]);
            add_row_high<W, HI, A + 1>(addr, na, q, old);
        }
    }
}

// Index j of 0 .. n-1 taken in the order 0, n-1, 1, n-2, ...: the tile
// columns near the uv origin (both ends of the wrapped axes), which hold the
// most entries, start first and do not trail the launch.
__device__ __forceinline__ int centre_first(int j, int n) { return (j & 1) ? n - 1 - (j >> 1) : (j >> 1); }

// Writes out the ring's slices (t-tiles) s in [from, to), when the ring holds
// planes [from TT, from TT + RP): a slice that the chunk owns and a footprint
// touched (tile_occ) goes to the stack, its planes past the ring's end as
// zeros (no footprint reached them).  With `clear`, each thread zeroes the
// ring cells it has just read, which leaves the slices' ring planes zero for
// the planes that take their slots: every other cell of those planes is zero
// already (a slice no footprint touched, or outside the chunk, received no
// contribution, and padding cells never do).
template <int W, int R, bool DET>
__device__ __forceinline__ void flush_slices(int from, int to, const Launch &L, int tv, int tu, int chunk_tt0,
                                             int chunk_ntt, const uint8_t *__restrict__ tile_occ, int scale,
                                             unsigned char *smem, float2 *__restrict__ stack, bool clear) {
    using Sm = GridSmem<W, R, DET>;
    constexpr int RP = Sm::RP, PS = Sm::PS;
    const int ring_end = from * TT + RP;
    const int last = min(to, from + (RP + TT - 1) / TT);
    const size_t plane = (size_t)L.Np * L.Np;
    for (int sl = max(from, chunk_tt0); sl < min(last, chunk_tt0 + chunk_ntt); ++sl) {
        if (!tile_occ[((size_t)sl * L.ntv + tv) * L.ntu + tu]) continue;
        // pairs of cells, ordered (plane, column block, row, pair) so that each
        // column block's R rows go out as one contiguous run
        for (int i = threadIdx.x; i < TT * R * TU / 2; i += kGridThreads) {
            const int pair = i & 1, lr = (i >> 1) % R, blk = (i / (2 * R)) % (TU / CB), pl = i / (TU * R / 2);
            const int lc = blk * CB + 2 * pair;
            const int t = sl * TT + pl;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (t < ring_end) {
                const int cell = (t % RP) * PS + lr * kRowPad + lc;
                if constexpr (DET) {
                    auto sum = [&](size_t ring, int c) {
                        unsigned *lo = reinterpret_cast<unsigned *>(smem + ring) + c, *hi = lo + Sm::HI / 4;
                        const long long q = (long long)((unsigned long long)*hi << 32 | *lo);
                        if (clear) *lo = *hi = 0u;
                        return ldexpf(__ll2float_rn(q), -scale);
                    };
                    v = make_float4(sum(Sm::re, cell), sum(Sm::im, cell), sum(Sm::re, cell + 1), sum(Sm::im, cell + 1));
                } else {
                    float *sre = reinterpret_cast<float *>(smem + Sm::re);
                    float *sim = reinterpret_cast<float *>(smem + Sm::im);
                    v = make_float4(sre[cell], sim[cell], sre[cell + 1], sim[cell + 1]);
                    if (clear) sre[cell] = sim[cell] = sre[cell + 1] = sim[cell + 1] = 0.f;
                }
            }
            float2 *dst = stack + (size_t)(t - chunk_tt0 * TT) * plane + tiled_index(tv * R + lr, tu * TU + lc, L.Np);
            *reinterpret_cast<float4 *>(dst) = v;
        }
    }
}

// DET: the deterministic mode (WS_FLAG_DETERMINISTIC).  The ring sums in 64-bit
// fixed point with one scale 2^scale for the CTA, chosen so that no sum can
// exceed 2^62: |sum| <= E max|V~| wbound for the column's E entries, wbound
// bounding |C_x C_y C_z|.  The scale depends only on the column's set of
// entries (all of them, whatever the chunk), and integer additions do not depend on
// their order, so the stack -- and the dirty image -- come out bit for bit the same
// whatever order the binning's atomics and the warps' schedule give the entries.
template <int W, int R, bool DET>
__global__ void __launch_bounds__(kGridThreads, grid_ctas_per_sm(W, R, DET))
grid3d_kernel(Launch L, const float *__restrict__ coef, int deg, const VisRec *__restrict__ rec,
              const uint32_t *__restrict__ offsets, const uint32_t *__restrict__ list,
              const uint8_t *__restrict__ tile_occ, int chunk_tt0, int chunk_ntt, float wbound,
              float2 *__restrict__ stack) {
    using Sm = GridSmem<W, R, DET>;
    constexpr int PS = Sm::PS, RP = Sm::RP, HI = Sm::HI, S = Sm::S, SP = Sm::SP, WX = Sm::WX;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned col_max;                      // DET: max |V~| of the column's entries (float bits)
    const int tu = centre_first(blockIdx.x % L.ntu, L.ntu);
    const int tv = centre_first(blockIdx.x / L.ntu, L.ntv);
    // the bins whose footprints reach the chunk's planes [plo, phi)
    const int k_lo = max(0, chunk_tt0 - (TT + W - 2) / TT), k_hi = chunk_tt0 + chunk_ntt;
    const int plo = chunk_tt0 * TT, phi = plo + chunk_ntt * TT;
    const uint32_t *__restrict__ off = offsets + ((size_t)tv * L.ntu + tu) * L.ntt;
    if (off[k_lo] == off[k_hi]) return;              // untouched column: the transforms treat it as zero
    const uint32_t all_beg = DET ? off[0] : 0u, all_end = DET ? off[L.ntt] : 0u;     // DET: the column's entries
    float *scoef = reinterpret_cast<float *>(smem + Sm::coef);
    {
        float4 *qre = reinterpret_cast<float4 *>(smem + Sm::re), *qim = reinterpret_cast<float4 *>(smem + Sm::im);
        for (int i = threadIdx.x; i < (int)(ring_bytes(W, R, DET) / 16); i += kGridThreads) {
            qre[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            qim[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    if constexpr (DET) {
        if (threadIdx.x == 0) col_max = 0u;
        __syncthreads();
        float m = 0.f;
        for (uint32_t e = all_beg + threadIdx.x; e < all_end; e += kGridThreads) {
            const VisRec r = rec[list[e]];
            m = fmaxf(m, fmaxf(fabsf(r.vre), fabsf(r.vim)));
        }
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0) atomicMax(&col_max, __float_as_uint(m));   // non-negative floats order as integers
    }
    // slot l < 3W is (axis l / W, tap l % W); coef holds the (u, v) table and
    // then the w table, W x (deg + 1) each; coefficients past deg are zero
    for (int i = threadIdx.x; i < S * kCoefStride; i += kGridThreads) {
        const int l = i / kCoefStride, m = i - l * kCoefStride, axis = l / W, tap = l - axis * W;
        const int row = (axis == 2 ? W : 0) + tap;
        scoef[i] = m <= deg ? coef[row * (deg + 1) + m] : 0.f;
    }
    __syncthreads();
    const int Np = L.Np;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u_org = tu * TU, v_org = tv * R;
    float *wts = reinterpret_cast<float *>(smem + Sm::wt) + warp * kChunk * SP;
    int4 *items = reinterpret_cast<int4 *>(smem + Sm::item) + warp * kChunk;
    float2 *vals = reinterpret_cast<float2 *>(smem + Sm::val) + warp * kChunk;
    float4 *nus = reinterpret_cast<float4 *>(smem + Sm::nu) + warp * kChunk;
    const unsigned re_base = (unsigned)__cvta_generic_to_shared(smem + Sm::re);
    const unsigned im_base = (unsigned)__cvta_generic_to_shared(smem + Sm::im);
    int scale = 0;                                   // DET: sums are kept as integers in units of 2^-scale
    if constexpr (DET) {
        const float bound = (float)(all_end - all_beg) * __uint_as_float(col_max) * wbound;
        if (bound > 0.f) {
            int ex;
            frexpf(bound, &ex);                          // bound < 2^ex
            scale = 62 - ex;
        }
    }
    // 2^scale in two factors that FP32 holds; the staged values are multiplied by it
    // (exactly), so a contribution needs no scaling of its own
    const float up0 = ldexpf(1.f, scale / 2), up1 = ldexpf(1.f, scale - scale / 2);
    int cur = -1;                                    // t-tile of the ring's first plane; -1: none yet
    for (int k = k_lo; k < k_hi; ++k) {
        const uint32_t beg = off[k], end = off[k + 1];
        if (beg == end) continue;
        if (cur >= 0) {
            // bin k reaches planes [k TT, k TT + RP): the ring's planes before k TT are final
            __syncthreads();
            flush_slices<W, R, DET>(cur, k, L, tv, tu, chunk_tt0, chunk_ntt, tile_occ, scale, smem, stack, true);
            __syncthreads();
        }
        cur = k;
        // this warp's share of the bin's entries
        const uint32_t E = end - beg;
        const uint32_t per = (E + kGridWarps - 1) / kGridWarps;
        const uint32_t wbeg = beg + min(E, warp * per), wend = beg + min(E, (warp + 1) * per);
        for (uint32_t cbeg = wbeg; cbeg < wend; cbeg += kChunk) {
            const int n = (int)min((uint32_t)kChunk, wend - cbeg);
            // 1. lane j: entry j's part of the footprint inside the column and the chunk's planes
            if (lane < n) {
                const uint32_t kv = list[cbeg + lane];
                const VisRec r = rec[kv];
                Span su[2], sv[2];
                const int nsu = tile_spans(u_org, r.r0, Np, W, TU, su[0], su[1]);
                const int nsv = tile_spans(v_org, r.s0, Np, W, R, sv[0], sv[1]);
                const int c0 = max(0, plo - r.t0), c1 = min(W, phi - r.t0);
                int4 it;
                const float2 V = DET ? make_float2(r.vre * up0 * up1, r.vim * up0 * up1) : make_float2(r.vre, r.vim);
                // (values that are not finite keep the conversion that saturates)
                const bool finite = !DET || (fabsf(V.x) <= 0x1p126f && fabsf(V.y) <= 0x1p126f);
                if (nsu == 1 && nsv == 1 && finite) {
                    const int na = su[0].a1 - su[0].a0, nb = sv[0].a1 - sv[0].a0, nc = max(c1 - c0, 0);
                    const int slot = (r.t0 + c0) % RP;      // ring slot of the part's first plane
                    it.x = (sv[0].a0 - sv[0].off) * kRowPad + (su[0].a0 - su[0].off);
                    it.y = na | nb << 4 | nc << 8 | su[0].a0 << 12 | sv[0].a0 << 16 | c0 << 20 | slot << 24;
                    it.z = __float_as_int(1.0f / (float)nb);
                } else {
                    it.x = 0;
                    it.y = kGeneral;
                    it.z = 0;
                }
                it.w = (int)kv;
                items[lane] = it;
                vals[lane] = V;
                nus[lane] = make_float4(r.nux, r.nuy, r.nuz, 0.f);
            }
            __syncwarp();
            // 2. the chunk's weights: pair q = (entry j, slot l), Horner from nu^16
            //    down; the u weights are kept from the part's first tap a0 on
            for (int q = lane; q < n * S; q += 32) {
                const int j = q / S, l = q - j * S, axis = l / W;
                const float4 nv = nus[j];
                const float nu = axis == 0 ? nv.x : (axis == 1 ? nv.y : nv.z);
                const float4 *c = reinterpret_cast<const float4 *>(scoef + l * kCoefStride);
                float acc = c[4].x;
#pragma unroll
                for (int b = 3; b >= 0; --b) {
                    const float4 c4 = c[b];
                    acc = fmaf(acc, nu, c4.w);
                    acc = fmaf(acc, nu, c4.z);
                    acc = fmaf(acc, nu, c4.y);
                    acc = fmaf(acc, nu, c4.x);
                }
                int pos = WX + l - W;
                if (axis == 0) {
                    const int y = items[j].y;
                    pos = l - (y == kGeneral ? 0 : (y >> 12) & 15);
                }
                if (pos >= 0) wts[j * SP + pos] = acc;
            }
            __syncwarp();
            // 3. add the chunk's entries one after the other
            for (int j = 0; j < n; ++j) {
                const int4 it = items[j];
                const float2 V = vals[j];
                const float *wt = wts + j * SP;
                if (it.y != kGeneral) {
                    const int na = it.y & 15, nb = (it.y >> 4) & 15, nc = (it.y >> 8) & 15;
                    const int b0 = (it.y >> 16) & 15, cw0 = (it.y >> 20) & 15;
                    const int slot0 = (it.y >> 24) & 31;
                    const float inv_nb = __int_as_float(it.z);
                    const int nbc = nb * nc;
                    // the part's u-tap weights (staged from its first tap on; those
                    // past na are not used), all read before the first reduction
                    float wx[WX];
#pragma unroll
                    for (int a4 = 0; a4 < WX / 4; ++a4) {
                        const float4 v = reinterpret_cast<const float4 *>(wt)[a4];
                        wx[4 * a4] = v.x;
                        wx[4 * a4 + 1] = v.y;
                        wx[4 * a4 + 2] = v.z;
                        wx[4 * a4 + 3] = v.w;
                    }
                    for (int q = lane; q < nbc; q += 32) {
                        // q = cc nb + bb, q < 144: (q + 1/2) / nb is at least 1/24 from an integer
                        const int cc = __float2int_rz(((float)q + 0.5f) * inv_nb), bb = q - cc * nb;
                        const float wyz = wt[WX + b0 + bb] * wt[WX + W + cw0 + cc];
                        int slot = slot0 + cc;
                        if (slot >= RP) slot -= RP;
                        const unsigned o = (unsigned)(it.x + slot * PS + bb * kRowPad) * 4;
                        if constexpr (DET) {
                            long long qre[W], qim[W];
                            unsigned ore[W], oim[W];
                            add_row_low<W, HI>(re_base + o, wx, na, V.x * wyz, qre, ore);
                            add_row_low<W, HI>(im_base + o, wx, na, V.y * wyz, qim, oim);
                            add_row_high<W, HI>(re_base + o, na, qre, ore);
                            add_row_high<W, HI>(im_base + o, na, qim, oim);
                        } else {
                            add_row<W>(re_base + o, wx, na, V.x * wyz);
                            add_row<W>(im_base + o, wx, na, V.y * wyz);
                        }
                    }
                } else {
                    // the part wraps around an axis (N' < W + R; or see above): every span pair, taps one by one
                    const VisRec r = rec[it.w];
                    Span su[2], sv[2];
                    const int nsu = tile_spans(u_org, r.r0, Np, W, TU, su[0], su[1]);
                    const int nsv = tile_spans(v_org, r.s0, Np, W, R, sv[0], sv[1]);
                    const int c0 = max(0, plo - r.t0), c1 = min(W, phi - r.t0);
                    for (int iu = 0; iu < nsu; ++iu)
                        for (int iv = 0; iv < nsv; ++iv) {
                            const int na = su[iu].a1 - su[iu].a0, nb = sv[iv].a1 - sv[iv].a0, nc = c1 - c0;
                            for (int q = lane; q < na * nb * nc; q += 32) {
                                const int a = su[iu].a0 + q % na, b = sv[iv].a0 + (q / na) % nb, c = c0 + q / (na * nb);
                                const float w = wt[a] * wt[WX + b] * wt[WX + W + c];
                                const unsigned o = (unsigned)(((r.t0 + c) % RP) * PS + (b - sv[iv].off) * kRowPad +
                                                              (a - su[iu].off)) * 4;
                                add_cell<DET, HI>(re_base + o, V.x * w);
                                add_cell<DET, HI>(im_base + o, V.y * w);
                            }
                        }
                }
            }
            __syncwarp();                              // the chunk's staging is read before the next overwrites it
        }
    }
    __syncthreads();
    flush_slices<W, R, DET>(cur, cur + (RP + TT - 1) / TT, L, tv, tu, chunk_tt0, chunk_ntt, tile_occ, scale, smem,
                            stack, false);
}

// ---------------------------------------------------------------------------
// Gridding in registers (W <= 9, 16-row tiles, FP32 sums in any order).
//
// A bin's footprints reach 16 planes (8 + W - 1 <= 16).  Each warp owns 4 x 8 of a
// tile's 16 x 16 cells and a lane one of them, with its sums of all 16 planes in
// registers, plane t in sum t mod 16: a t-tile's planes are sums 0..7 or 8..15, and
// moving on to the next bin writes out and clears one half.  There is no ring in
// shared memory, and there are no atomics.
//
// The CTA stages the column's entries kRegEntries at a time, whatever their bins: per
// entry its weights at the tile's 16 columns and 16 rows and at 16 planes, zero where
// the footprint does not reach.  (A chunk per bin, 11 entries at the median, spent
// most of its instructions on the staging's fixed part.)  A warp then takes only the
// entries that touch its cells (29 % of a tile's for W = 7): a lane forms C_x C_y V
// for its cell once and adds C_z C_x C_y V to its 16 sums, one packed multiply-add
// for both components of a plane.
//
// Every product and sum is FP32, as in grid3d_kernel.  The same contraction on the
// tensor cores (mma.m16n8k8, each factor split into two TF32 terms) took 6.63 ms on the
// survey (18.9 M entries) where this takes 5.29 and grid3d_kernel 9.8, and was less exact:
// 1.92e-7 from an FP64 plan where these two stay at 1.64e-7 (1,000 visibilities, N = 256,
// W = 7), and values near 2^-115 lost digits, their low terms below the tensor core's smallest.
// (The 80 registers that three CTAs an SM allow spill 32 bytes in the staging, 64 for W <= 4.)
constexpr int kRegMaxW = TT + 1;
constexpr int kRegEntries = 64;                    // staged per chunk
constexpr int kRegStride = 60;                     // floats per staged entry: weights read as float4
constexpr int kRegMaxBins = 520;                   // t-tiles of a column: |t| < 2040, 8 planes each, and two more
enum : int { kEntU = 0, kEntV = 16, kEntT = 32, kEntVal = 48, kEntOff = 50, kEntNu = 51 };

// Cells 0..15 of a tile axis that a footprint starting `off` cells after the
// tile's origin (mod n) covers, as bits.
__device__ __forceinline__ unsigned axis_mask(int off, int n, int W) {
    const unsigned taps = (1u << W) - 1u;
    unsigned m = off < 16 ? taps << off : 0u;
    if (off + W > n) m |= taps >> (n - off);
    return m & 0xffffu;
}

template <int W>
__global__ void __launch_bounds__(kGridThreads, 3)
grid3d_cells_kernel(Launch L, const float *__restrict__ coef, int deg, const VisRec *__restrict__ rec,
                    const uint32_t *__restrict__ offsets, const uint32_t *__restrict__ list,
                    const uint8_t *__restrict__ tile_occ, int chunk_tt0, int chunk_ntt, float2 *__restrict__ stack) {
    static_assert(W <= kRegMaxW, "a bin's footprints stay within 16 planes");
    __shared__ __align__(16) float ents[2][kRegEntries * kRegStride];
    __shared__ unsigned masks[2][kRegEntries];     // the entries' cells: columns in bits 0..15, rows in 16..31
    __shared__ __align__(16) float scoef[3 * W * kCoefStride];
    __shared__ uint32_t soff[kRegMaxBins];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Np = L.Np;
    const int tu = centre_first(blockIdx.x % L.ntu, L.ntu);
    const int tv = centre_first(blockIdx.x / L.ntu, L.ntv);
    const int u_org = tu * TU, v_org = tv * 16;
    // the bins whose footprints reach the chunk's planes
    const int k_lo = max(0, chunk_tt0 - (TT + W - 2) / TT), k_hi = chunk_tt0 + chunk_ntt;
    const uint32_t *__restrict__ off = offsets + ((size_t)tv * L.ntu + tu) * L.ntt;
    uint32_t pos = off[k_lo];
    const uint32_t all_end = off[k_hi];
    if (pos == all_end) return;                      // untouched column: the transforms treat it as zero
    for (int i = tid; i <= k_hi - k_lo; i += kGridThreads) soff[i] = off[k_lo + i];
    for (int i = tid; i < 3 * W * kCoefStride; i += kGridThreads) {
        const int l = i / kCoefStride, m = i - l * kCoefStride, axis = l / W;
        scoef[i] = m <= deg ? coef[((axis == 2 ? W : 0) + l - axis * W) * (deg + 1) + m] : 0.f;
    }
    __syncthreads();

    // lanes 0..7 of a warp hold the records of entries warp + 8 lane of the next chunk
    VisRec r{};
    auto fetch = [&] {
        const uint32_t p = pos + warp + kGridWarps * lane;
        if (lane < kRegEntries / kGridWarps && p < all_end) r = rec[list[p]];
    };
    fetch();
    const int row0 = 4 * (warp >> 1), col0 = 8 * (warp & 1);         // this warp's cells
    const int row = row0 + (lane >> 3), col = col0 + (lane & 7);     // this lane's
    const unsigned my_cells = (0xffu << col0) | (0xfu << (16 + row0));
    float2 c[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) c[i] = make_float2(0.f, 0.f);
    const size_t plane = (size_t)Np * Np;
    // writes out t-tile s, if the chunk owns it, and zeroes its sums
    auto flush = [&](int s, bool touched) {
        float2 *dst = stack + (size_t)(s - chunk_tt0) * TT * plane + tiled_index(v_org + row, u_org + col, Np);
        const bool own = touched && s >= chunk_tt0 && s < k_hi;
        auto half = [&](int first) {
#pragma unroll
            for (int i = 0; i < TT; ++i) {
                if (own) dst[i * plane] = c[first + i];
                c[first + i] = make_float2(0.f, 0.f);
            }
        };
        if (s & 1)
            half(8);
        else
            half(0);
    };
    // the planes past bin k's t-tile, where some footprint of the bin or the bins before may have reached
    auto flush_next = [&](int s) { flush(s, s < k_hi && tile_occ[((size_t)s * L.ntv + tv) * L.ntu + tu]); };
    const int axis = lane / W < 3 ? lane / W : 2, tap = lane - axis * W;     // staging: this lane's weight slot
    const int off_shift = 13 * axis, axis_len = axis == 2 ? 16 : Np, axis_base = 16 * axis;
    const unsigned off_mask = axis == 2 ? 15u : 0x1fffu;
    int k = k_lo, cur = -1, buf = 0;
    while (pos < all_end) {
        const int n = (int)min((uint32_t)kRegEntries, all_end - pos);
        float *ent = ents[buf];
        // 1. staging: this warp's entries warp, warp + 8, ...
        const int mine = n > warp ? (n - warp + kGridWarps - 1) / kGridWarps : 0;
        if (lane < mine) {
            float *e = ent + (warp + kGridWarps * lane) * kRegStride;
            int du = r.r0 - u_org, dv = r.s0 - v_org;
            if (du < 0) du += Np;
            if (dv < 0) dv += Np;
            e[kEntVal] = r.vre;
            e[kEntVal + 1] = r.vim;
            masks[buf][warp + kGridWarps * lane] = axis_mask(du, Np, W) | axis_mask(dv, Np, W) << 16;
            e[kEntNu] = r.nux;
            e[kEntNu + 1] = r.nuy;
            e[kEntNu + 2] = r.nuz;
            e[kEntOff] = __int_as_float(du | dv << 13 | (r.t0 & 15) << 26);
        }
        for (int i = 0; i < mine; i += 2) {            // zero the weights: 16 lanes an entry
            const int j = i + (lane >> 4);
            if (j < mine && (lane & 15) < 12)
                *reinterpret_cast<float4 *>(ent + (warp + kGridWarps * j) * kRegStride + 4 * (lane & 15)) =
                    make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncwarp();
        if (mine > 0 && lane < 3 * W) {
            float cf[17];
            const float4 *c4 = reinterpret_cast<const float4 *>(scoef + lane * kCoefStride);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float4 v = c4[b];
                cf[4 * b] = v.x;
                cf[4 * b + 1] = v.y;
                cf[4 * b + 2] = v.z;
                cf[4 * b + 3] = v.w;
            }
            cf[16] = c4[4].x;
            for (int i = 0; i < mine; i += 2) {        // Horner from nu^16 down, two entries at a time
                float *e0 = ent + (warp + kGridWarps * i) * kRegStride;
                float *e1 = i + 1 < mine ? e0 + kGridWarps * kRegStride : e0;
                const float2 nu = make_float2(e0[kEntNu + axis], e1[kEntNu + axis]);
                float2 w = dup2(cf[16]);
#pragma unroll
                for (int b = 15; b >= 0; --b) {        // (a packed step would have to copy each coefficient)
                    w.x = fmaf(w.x, nu.x, cf[b]);
                    w.y = fmaf(w.y, nu.y, cf[b]);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {          // the same steps for every axis: no divergence
                    float *e = h ? e1 : e0;
                    int p = (int)((__float_as_uint(e[kEntOff]) >> off_shift) & off_mask) + tap;
                    if (p >= axis_len) p -= axis_len;
                    if (p < 16) e[axis_base + p] = h ? w.y : w.x;
                }
            }
        }
        // the other buffer's readers are past this barrier before anyone stages into it again
        __syncthreads();
        const uint32_t chunk0 = pos;
        pos += n;
        fetch();
        // the chunk's bins one after the other; from here on the warps go their own way
        for (uint32_t b0 = chunk0; b0 < pos;) {
            while (soff[k + 1 - k_lo] == b0) ++k;                            // bins with nothing left
            const uint32_t b1 = min(pos, soff[k + 1 - k_lo]);
            // 2. the window moves to bin k: planes it has left behind are final
            if (k != cur) {
                if (cur >= 0) {
                    flush(cur, true);
                    if (k > cur + 1) flush_next(cur + 1);
                }
                cur = k;
            }
            // 3. the entries that touch this warp's cells, one after the other
            for (int b = (int)(b0 - chunk0); b < (int)(b1 - chunk0); b += 32) {
                bool hit = false;
                if (b + lane < (int)(b1 - chunk0)) {
                    const unsigned m = masks[buf][b + lane] & my_cells;
                    hit = (m & 0xffffu) && (m >> 16);
                }
                for (unsigned hits = __ballot_sync(0xffffffffu, hit); hits; hits &= hits - 1u) {
                    const float *e = ent + (b + __ffs(hits) - 1) * kRegStride;
                    const float2 V = *reinterpret_cast<const float2 *>(e + kEntVal);
                    const float2 p = mul2(V, dup2(e[kEntU + col] * e[kEntV + row]));
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 z = *reinterpret_cast<const float4 *>(e + kEntT + 4 * q);
                        c[4 * q] = fma2(dup2(z.x), p, c[4 * q]);
                        c[4 * q + 1] = fma2(dup2(z.y), p, c[4 * q + 1]);
                        c[4 * q + 2] = fma2(dup2(z.z), p, c[4 * q + 2]);
                        c[4 * q + 3] = fma2(dup2(z.w), p, c[4 * q + 3]);
                    }
                }
            }
            b0 = b1;
        }
        buf ^= 1;
    }
    flush(cur, true);
    flush_next(cur + 1);
}

// Section 5.4: a visibility with w < 0 was degridded at -(u, v, w); the real
// sky's visibility at (u, v, w) is the conjugate of that.
__global__ void unfold_kernel(const double *__restrict__ uvw, int64_t M, float2 *__restrict__ vis) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    if (uvw[3 * k + 2] < 0.0) vis[k].y = -vis[k].y;
}

// ---------------------------------------------------------------------------
constexpr int kDegridThreads = 256;

// Degridding: Algorithm 6 steps 4-5.  One warp per visibility; lanes over the
// W x W (a, b) columns of the footprint (W^2 / 32 rounded up per lane), W planes
// each.  All of a lane's gathers are issued before any is used, so a warp keeps
// up to 2 W loads in flight.  Each chunk adds its planes' share to vis, in chunk order.
//
// The kernel waits for its gathers, and they share the L1's data pipe with the
// weights.  So a CTA takes up to kDegridRun x 8 consecutive visibilities of the
// tile-sorted list at a time: their footprints overlap and meet in its L1 (with
// consecutive visibilities dealt to different SMs, each SM fetched the same lines).
// The polynomial table sits in shared memory coefficient by coefficient, so a
// step of Horner's rule reads consecutive words, and the steps start at the
// table's degree.  A warp has the next visibility's record under way while it
// works on one.
constexpr int kDegridRun = 8;

template <int W>
__global__ void __launch_bounds__(kDegridThreads, W <= 5 ? 5 : (W <= 7 ? 4 : W <= 8 ? 3 : 1))
degrid3d_kernel(Launch L, const float *__restrict__ coef, int deg, const VisRec *__restrict__ rec,
                const uint32_t *__restrict__ order, const uint32_t *__restrict__ n_order,
                const float2 *__restrict__ stack, int plane0, int planes, float2 *__restrict__ vis) {
    constexpr int kPasses = (W * W + 31) / 32, kWarps = kDegridThreads / 32, S = 3 * W;
    __shared__ float swt[kWarps][S];
    __shared__ float scoef[(kMaxDeg + 1) * S];              // [m][u taps, v taps, w taps]
    for (int i = threadIdx.x; i < (deg + 1) * S; i += kDegridThreads) {
        const int m = i / S, l = i - m * S;
        scoef[i] = coef[(l < W ? l : l - W) * (deg + 1) + m];   // rows: the (u, v) table, then the w table
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = (int64_t)*n_order;                   // entries of the sorted list (dropped ones excluded)
    const int Np = L.Np;
    const size_t plane = (size_t)Np * Np;
    float *wt = swt[warp];
    // visibilities per warp and run: short runs while there are too few to go round
    const int64_t nwarps = (int64_t)gridDim.x * kWarps;
    const int run = (int)max((int64_t)1, min((int64_t)kDegridRun, n / (4 * nwarps)));
    for (int64_t base = (int64_t)blockIdx.x * kWarps * run; base < n; base += nwarps * run) {
        const int mine = (int)max((int64_t)0, min((int64_t)run, (n - base - warp + kWarps - 1) / kWarps));
        uint32_t ids = 0;                                   // lane i: this warp's i-th visibility
        if (lane < mine) ids = order[base + warp + kWarps * lane];
        VisRec next{};
        if (mine > 0) next = rec[__shfl_sync(0xffffffffu, ids, 0)];
        for (int i = 0; i < mine; ++i) {
            const uint32_t k = __shfl_sync(0xffffffffu, ids, i);
            const VisRec r = next;
            if (i + 1 < mine) next = rec[__shfl_sync(0xffffffffu, ids, i + 1)];
            if (r.t0 < 0) continue;
            const int c_lo = max(0, plane0 - r.t0);
            const int c_hi = min(W - 1, plane0 + planes - 1 - r.t0);
            if (c_lo > c_hi) continue;
            const int64_t t_rel = (int64_t)r.t0 - plane0;       // stack plane of tap c is t_rel + c
            const bool all_planes = c_lo == 0 && c_hi == W - 1; // uniform: the whole footprint is in the chunk
            float2 f[kPasses][W];
#pragma unroll
            for (int ps = 0; ps < kPasses; ++ps) {
                const int pair = lane + 32 * ps;
                const int a = pair % W, b = pair / W;
                const bool live = pair < W * W;
                const float2 *cell = stack + tiled_index(wrap_add(r.s0, live ? b : 0, Np), wrap_add(r.r0, a, Np), Np) +
                                     t_rel * (int64_t)plane;
                if (all_planes) {
#pragma unroll
                    for (int c = 0; c < W; ++c)
                        f[ps][c] = live ? __ldg(cell + (size_t)c * plane) : make_float2(0.f, 0.f);
                } else {
#pragma unroll
                    for (int c = 0; c < W; ++c) {
                        f[ps][c] = make_float2(0.f, 0.f);
                        if (live && c >= c_lo && c <= c_hi) f[ps][c] = __ldg(cell + (int64_t)c * (int64_t)plane);
                    }
                }
            }
            __syncwarp();                                       // the previous visibility's weights are read
            for (int l = lane; l < S; l += 32) {                // S > 32 for W >= 11
                const float nu = l < W ? r.nux : (l < 2 * W ? r.nuy : r.nuz);
                float acc = 0.f;                                // Horner from nu^deg down
#pragma unroll
                for (int m = kMaxDeg; m >= 0; --m)
                    if (m <= deg) acc = fmaf(acc, nu, scoef[m * S + l]);
                wt[l] = acc;
            }
            __syncwarp();
            float ar = 0.f, ai = 0.f;
#pragma unroll
            for (int ps = 0; ps < kPasses; ++ps) {
                const int pair = lane + 32 * ps;
                if (pair >= W * W) break;
                const int a = pair % W, b = pair / W;
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < W; ++c) s = fma2(dup2(wt[2 * W + c]), f[ps][c], s);
                const float wab = wt[a] * wt[W + b];
                ar = fmaf(wab, s.x, ar);
                ai = fmaf(wab, s.y, ai);
            }
            for (int o = 16; o > 0; o >>= 1) {
                ar += __shfl_xor_sync(0xffffffffu, ar, o);
                ai += __shfl_xor_sync(0xffffffffu, ai, o);
            }
            if (lane == 0) {
                float2 out = vis[k];
                out.x += ar * r.vre - ai * r.vim;
                out.y += ar * r.vim + ai * r.vre;
                vis[k] = out;
            }
        }
    }
}

inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
cudaError_t launch_prep(const ws_plan_s *p, const double *uvw, int64_t M, cudaStream_t s) {
    if (M == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)std::min<int64_t>(blocks_for(M, 256), (int64_t)p->sms * 8);
    prep_kernel<kPrepOnly><<<blocks, 256, 0, s>>>(p->L, uvw, nullptr, M, p->d_rec, p->d_drop, nullptr, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_clear_bins(const ws_plan_s *p, unsigned long long *drop, cudaStream_t s) {
    const int64_t n = p->ntiles + 1;
    const unsigned blocks = (unsigned)std::min<int64_t>(blocks_for(n, 256), (int64_t)p->sms * 8);
    clear_bins_kernel<<<blocks, 256, 0, s>>>(p->d_counts, n, p->d_tile_occ, p->ntiles, p->d_col_occ,
                                             (int64_t)p->L.ntt * p->L.ntu, drop);
    return cudaGetLastError();
}

cudaError_t launch_prep_count(const ws_plan_s *p, const double *uvw, const float2 *vis, int64_t M, bool grid,
                              float2 *zeroed, cudaStream_t s) {
    if (M == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)std::min<int64_t>(blocks_for(M, 256), (int64_t)p->sms * 8);
    if (grid)
        prep_kernel<kPrepGrid><<<blocks, 256, 0, s>>>(p->L, uvw, vis, M, p->d_rec, p->d_drop, p->d_counts,
                                                      p->d_tile_occ, nullptr);
    else
        prep_kernel<kPrepDegrid><<<blocks, 256, 0, s>>>(p->L, uvw, nullptr, M, p->d_rec, p->d_drop, p->d_counts,
                                                        p->d_tile_occ, zeroed);
    return cudaGetLastError();
}

cudaError_t launch_bound_grid_records(const ws_plan_s *p, const double *uvw, const float2 *vis, int64_t M,
                                      cudaStream_t s) {
    if (M == 0) return cudaSuccess;
    bound_grid_records_kernel<<<blocks_for(M, 256), 256, 0, s>>>(p->L, uvw, vis, M, p->d_brec, p->d_rec);
    return cudaGetLastError();
}

cudaError_t launch_count(const ws_plan_s *p, int64_t M, bool grid, cudaStream_t s) {
    cudaError_t e = launch_clear_bins(p, nullptr, s);
    if (e != cudaSuccess || M == 0) return e;
    if (grid)
        count_kernel<true><<<blocks_for(M, 256), 256, 0, s>>>(p->L, p->d_rec, M, p->d_counts, p->d_tile_occ);
    else
        count_kernel<false><<<blocks_for(M, 256), 256, 0, s>>>(p->L, p->d_rec, M, p->d_counts, p->d_tile_occ);
    return cudaGetLastError();
}

int sort_launches(const ws_plan_s *p, int64_t M) { return (p->ntiles + 1 > kScanPerBlock ? 3 : 1) + (M > 0 ? 1 : 0); }

cudaError_t launch_sort(const ws_plan_s *p, int64_t M, bool grid, cudaStream_t s) {
    const int64_t n = p->ntiles + 1;
    const int nb = (int)((n + kScanPerBlock - 1) / kScanPerBlock);
    scan_block_kernel<<<nb, kScanThreads, 0, s>>>(p->d_counts, p->d_offsets, p->d_blocksums, n);
    if (nb > 1) {                                // one block's scan is the whole one
        scan_sums_kernel<<<1, kScanThreads, 0, s>>>(p->d_blocksums, nb);
        scan_add_kernel<<<blocks_for(n, 256), 256, 0, s>>>(p->d_offsets, p->d_counts, p->d_blocksums, n);
    }
    if (M == 0) return cudaGetLastError();
    const unsigned vis_blocks = blocks_for(M, 256), blocks = vis_blocks + blocks_for(p->ntiles, 256);
    if (grid)
        scatter_kernel<true><<<blocks, 256, 0, s>>>(p->L, p->d_rec, M, (int)vis_blocks, p->d_counts, p->d_list,
                                                    p->d_tile_occ, p->ntiles, p->d_col_occ);
    else
        scatter_kernel<false><<<blocks, 256, 0, s>>>(p->L, p->d_rec, M, (int)vis_blocks, p->d_counts, p->d_list,
                                                     p->d_tile_occ, p->ntiles, p->d_col_occ);
    return cudaGetLastError();
}

cudaError_t launch_occ_count(const ws_plan_s *p, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(p->d_occ_counts, 0, (size_t)2 * p->L.ntt * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    occ_count_kernel<<<p->L.ntt, 256, 0, s>>>(p->L, p->d_tile_occ, p->d_col_occ, p->d_occ_counts);
    return cudaGetLastError();
}

cudaError_t launch_grid_chunk(const ws_plan_s *p, int chunk, int planes, cudaStream_t s) {
    const int chunk_tt0 = chunk * (p->P / TT), chunk_ntt = planes / TT;
    const unsigned nblocks = (unsigned)p->L.ntu * p->L.ntv;      // one CTA per tile column
    if (chunk_ntt == 0) return cudaSuccess;
    const int R = p->L.tv;
    const bool det = (p->flags & WS_FLAG_DETERMINISTIC) != 0;
    auto go = [&](auto kernel, size_t smem) -> cudaError_t {
        if (smem > kMaxGridSmem) return cudaErrorInvalidValue;   // set_tile_rows keeps this from happening
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kernel<<<nblocks, kGridThreads, smem, s>>>(p->L, p->d_wcoef, p->wdeg, p->d_rec, p->d_offsets, p->d_list,
                                                   p->d_tile_occ, chunk_tt0, chunk_ntt, p->wbound, p->d_stack);
        return cudaGetLastError();
    };
    // 16-row tiles of widths up to 9 keep their sums in registers; wider footprints reach
    // past the 16 planes that a lane holds, and taller tiles and the deterministic mode
    // keep their sums in shared memory
    auto cells = [&](auto kernel) -> cudaError_t {
        kernel<<<nblocks, kGridThreads, 0, s>>>(p->L, p->d_wcoef, p->wdeg, p->d_rec, p->d_offsets, p->d_list,
                                                p->d_tile_occ, chunk_tt0, chunk_ntt, p->d_stack);
        return cudaGetLastError();
    };
    auto width = [&](auto wc) -> cudaError_t {
        constexpr int w = decltype(wc)::value;
        if (det) {
            if (R == 16) return go(grid3d_kernel<w, 16, true>, GridSmem<w, 16, true>::bytes);
            if (R == 64) return go(grid3d_kernel<w, 64, true>, GridSmem<w, 64, true>::bytes);
            return go(grid3d_kernel<w, 32, true>, GridSmem<w, 32, true>::bytes);
        }
        if (R == 64) return go(grid3d_kernel<w, 64, false>, GridSmem<w, 64, false>::bytes);
        if (R == 32) return go(grid3d_kernel<w, 32, false>, GridSmem<w, 32, false>::bytes);
        if constexpr (w <= kRegMaxW)
            return cells(grid3d_cells_kernel<w>);
        else
            return go(grid3d_kernel<w, 16, false>, GridSmem<w, 16, false>::bytes);
    };
    switch (p->L.W) {
        case 1: return width(std::integral_constant<int, 1>{});
        case 2: return width(std::integral_constant<int, 2>{});
        case 3: return width(std::integral_constant<int, 3>{});
        case 4: return width(std::integral_constant<int, 4>{});
        case 5: return width(std::integral_constant<int, 5>{});
        case 6: return width(std::integral_constant<int, 6>{});
        case 7: return width(std::integral_constant<int, 7>{});
        case 8: return width(std::integral_constant<int, 8>{});
        case 9: return width(std::integral_constant<int, 9>{});
        case 10: return width(std::integral_constant<int, 10>{});
        case 11: return width(std::integral_constant<int, 11>{});
        case 12: return width(std::integral_constant<int, 12>{});
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_unfold(const ws_plan_s *p, const double *uvw, int64_t M, float2 *vis, cudaStream_t s) {
    (void)p;
    if (M == 0) return cudaSuccess;
    unfold_kernel<<<blocks_for(M, 256), 256, 0, s>>>(uvw, M, vis);
    return cudaGetLastError();
}

cudaError_t launch_degrid_chunk(const ws_plan_s *p, int chunk, int planes, int64_t M, float2 *vis,
                                cudaStream_t s) {
    if (M == 0) return cudaSuccess;
    // resident CTAs only (the kernel loops over the visibilities), at most one warp per visibility
    const int64_t want = blocks_for(M * 32, kDegridThreads);
    // CTAs per SM by (device, W), looked up once: the plan's device is current here
    auto resident = [&](auto kernel, int w) {
        constexpr int kDevices = 64;
        static std::atomic<int> per_sm[kDevices][kMaxW + 1];
        int b = p->dev >= 0 && p->dev < kDevices ? per_sm[p->dev][w].load(std::memory_order_relaxed) : 0;
        if (b == 0) {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kDegridThreads, 0) != cudaSuccess || b < 1)
                b = 1;
            if (p->dev >= 0 && p->dev < kDevices) per_sm[p->dev][w].store(b, std::memory_order_relaxed);
        }
        return (unsigned)std::min<int64_t>(want, (int64_t)p->sms * b);
    };
#define WS_DEGRID_CASE(w)                                                                                     \
    case w:                                                                                                  \
        degrid3d_kernel<w><<<resident(degrid3d_kernel<w>, w), kDegridThreads, 0, s>>>(                       \
            p->L, p->d_wcoef, p->wdeg, p->d_rec, p->d_list, p->d_offsets + p->ntiles, p->d_stack, chunk * p->P, \
            planes, vis);                                                                                    \
        break;
    switch (p->L.W) {
        WS_DEGRID_CASE(1)
        WS_DEGRID_CASE(2)
        WS_DEGRID_CASE(3)
        WS_DEGRID_CASE(4)
        WS_DEGRID_CASE(5)
        WS_DEGRID_CASE(6)
        WS_DEGRID_CASE(7)
        WS_DEGRID_CASE(8)
        WS_DEGRID_CASE(9)
        WS_DEGRID_CASE(10)
        WS_DEGRID_CASE(11)
        WS_DEGRID_CASE(12)
        default:
            return cudaErrorInvalidValue;
    }
#undef WS_DEGRID_CASE
    return cudaGetLastError();
}

}  // namespace ws
