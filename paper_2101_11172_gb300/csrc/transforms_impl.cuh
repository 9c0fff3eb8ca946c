// Kernel templates of the fused plane transforms (see transforms.cu).
//
// NP selects the FFT code: 0 = the runtime plan (any N'); 512, 1024, 2048, 4096
// = the compile-time plans of fft.cuh.  Each translation unit instantiates
// Transforms<NP> for its sizes.
#pragma once

#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fft.cuh"
#include "ws_internal.hpp"

namespace ws {
namespace tf {

constexpr int kPerCta = 2;          // columns per CTA of the column kernels
// Whether N' has a compile-time plan.
inline bool compile_time_size(int Np) { return Np == 512 || Np == 1024 || Np == 2048 || Np == 4096; }
// CTA sizes follow the transform: N'/16 threads for a row and twice that for a
// pair of columns, one radix-16 butterfly per thread in a stage (two at N' =
// 4096 for the columns).  With 256 threads at every size most of a CTA idled on
// short rows (N' = 512: 32 butterflies in the first stage).  Runtime plans
// bring their own (FftPlan::row_threads, col_threads).  The minimum of resident
// CTAs bounds the registers: 128 a thread for rows and runtime plans, 80 for columns.
// (Rows at 80 registers and three CTAs of 256 threads per SM, with one row buffer
// and z read from global memory to fit, were slower: inv_rows 13.6 against 9.5 ms and
// fwd_rows 9.2 against 8.6 on 366 planes of N' = 4096.)
template <int NP>
WS_HD constexpr int row_threads_max() {
    return NP ? NP / 16 : kMaxFftThreads;
}
template <int NP>
WS_HD constexpr int col_threads_max() {
    return NP ? (NP > 2048 ? 128 : NP / 8) : kMaxFftThreads;
}
template <int NP>
WS_HD constexpr int row_ctas() {
    return NP ? 512 / row_threads_max<NP>() : 2;
}
template <int NP>
WS_HD constexpr int col_ctas() {
    return NP == 4096 ? 3 : NP ? 768 / col_threads_max<NP>() : 2;
}
// Row CTAs that an SM can hold by threads and registers, and the shared memory
// that each may have for `ctas` of them to fit (228 KB per SM, 1 KB of it reserved per CTA).
inline int row_threads_of(const FftPlan &F) { return compile_time_size(F.n) ? F.n / 16 : F.row_threads; }
inline int row_cta_limit(const FftPlan &F) { return 512 / row_threads_of(F); }
inline size_t cta_smem(int ctas) { return (size_t)228 * 1024 / ctas - 1024; }

// The crop index of grid index g (0 <= g < N'): below N = 2 half inside the centred
// crop, at least N outside it.  One minimum for both: g + half - N' wraps to a huge
// value unless g is in the grid's last half columns.
__device__ __forceinline__ unsigned grid_to_crop(int g, int half, int Np) {
    const unsigned c = (unsigned)(g + half);
    return min(c, c - (unsigned)Np);
}

// The column kernels' transforms (two columns).  PRUNE (fftst::PRUNE_IN /
// PRUNE_OUT, compile-time plans with N' = 2N only): the inputs outside the
// centred half are zero / the outputs outside it are not wanted, and the
// transform skips them.
template <int NP, bool INV, int PRUNE, class Load, class Store>
__device__ __forceinline__ void column_fft(float2 *buf, const FftPlan &F, const float2 *__restrict__ tw, Load load,
                                           Store store) {
    if constexpr (NP == 0)
        fft_many<kPerCta, INV>(buf, F, tw, threadIdx.x, blockDim.x, load, store);
    else if constexpr (NP == 4096)
        fft_4096_two_stage<kPerCta, PRUNE>(buf, tw + F.bases[1], INV, threadIdx.x, load, store);
    else
        fft_static<NP, kPerCta, col_threads_max<NP>(), PRUNE>(buf, tw, INV, threadIdx.x, load, store);
}

// Calls f(m) for the elements of a butterfly of R that count: all of them, or the first and last quarter.
template <int R, bool PRUNED, class F>
__device__ __forceinline__ void for_live(F f) {
#pragma unroll
    for (int m = 0; m < R; ++m)
        if (!PRUNED || m < R / 4 || m >= 3 * R / 4) f(m);
}
template <class A>
__device__ __forceinline__ constexpr int length_of() {
    return (int)std::extent<std::remove_reference_t<A>>::value;
}

// The twiddle bases a row kernel's thread keeps across planes.
struct NoRowTw {
    __device__ __forceinline__ NoRowTw(const float2 *, bool, int) {}
};
template <int NP>
struct RowTwOf {
    using type = fftst::RowTw<NP, NP / 16>;
};
template <>
struct RowTwOf<0> {
    using type = NoRowTw;
};

// CROP: N' = 2N on a compile-time plan, so the crop is exactly the centred half.
template <int NP>
inline bool crop_half(const Launch &L) { return NP >= 512 && 2 * L.N == L.Np; }

// -- degridding --------------------------------------------------------------

// g times e, the screened value one plane on, with the products rounded in a fixed
// order: (g.x e.x - g.y e.y, g.y e.x + g.x e.y), those with e.y first.
__device__ __forceinline__ float2 step_screen(float2 g, float2 e) {
    return fma2(g, dup2(e.x), mul2(swap2(g), make_float2(-e.y, e.y)));
}

// Planes per exact evaluation of the screen in fwd_rows: in between, each
// pixel's screened value advances one plane by a product with exp(-2 pi i z).
constexpr int kScreenSteps = 8;

// One CTA owns image row ii for a run of planes.
//
// STEP (fwd_rows_step): shared memory keeps the screened row g = row x exp(-2 pi i
// t z) and the step exp(-2 pi i z), so each plane costs the step, one FFT and the
// stores of the strips some footprint reads.  g is evaluated exactly on every
// kScreenSteps-th plane of the CTA's share; on the planes between, the FFT's first
// stage reads g and leaves g x step in its place for the next plane.  Each pixel is
// read by the same thread on every plane, so the update needs no barrier.  The exact
// evaluations read the corrected row and its z from shared memory too (keep_rows),
// or, where that would cost a resident CTA, from global memory.
//
// Otherwise shared memory keeps the row and half a row of z and of the plane's
// screen, evaluated exactly on every plane as in inv_rows: the N/2 + 1 screens that
// a pixel and its mirror image share.  That takes the room of STEP's two rows.
// Stepping these sizes too (N above about 2400) took 29.4 instead of 30.0 ms at N = 4096
// (282 planes) but moved the error against the exact DFT: 2.07e-7 -> 2.35e-7 at N = 2560.
template <int NP, bool CROP, bool STEP>
__global__ void __launch_bounds__(row_threads_max<NP>(), row_ctas<NP>())
fwd_rows_kernel(Launch L, FftPlan F, const float2 *__restrict__ tw, const float2 *__restrict__ img,
                const float *__restrict__ corr, const float2 *__restrict__ zsplit,
                const uint8_t *__restrict__ col_occ, int plane0, int planes, int keep_rows,
                float2 *__restrict__ stack) {
    extern __shared__ __align__(16) float2 sbuf[];
    const int Np = L.Np, N = L.N, half = N / 2;
    float2 *grow = sbuf + F.stride;                              // N: the screened row (16-byte aligned)
    float2 *erow = grow + N;                                     // N: exp(-2 pi i z)
    float2 *irow = STEP ? erow + N : grow;                       // N if keep_rows
    float2 *zrow = irow + N;                                     // N if keep_rows
    float2 *scr = irow + N;                                      // N/2 + 1 unless STEP: exp(2 pi i t z)
    float2 *zhalf = scr + N / 2 + 1;                             // N/2 + 1 unless STEP: z
    uint8_t *occ = reinterpret_cast<uint8_t *>(STEP ? erow + (keep_rows ? 3 : 1) * N
                                                    : zhalf + N / 2 + 1);   // ntu: strips of the current t-tile
    const int ii = blockIdx.x, tid = threadIdx.x, T = NP ? row_threads_max<NP>() : (int)blockDim.x;
    // this CTA's planes: an equal share of the chunk's valid planes
    const int nvalid = min(planes, L.Nw - plane0);
    const int per = (nvalid + (int)gridDim.y - 1) / (int)gridDim.y;
    const int p_begin = (int)blockIdx.y * per, p_end = min(nvalid, p_begin + per);
    if (p_begin >= p_end) return;
    const size_t pix0 = (size_t)ii * N;
    // Algorithm 6 step 2, image x h_x h_y h_z (a real-sky plan reads only the image's real part)
    auto corrected = [&](int jj) {
        const float h = corr[pix0 + jj];
        const float2 f = img[pix0 + jj];
        return make_float2(h * f.x, L.fold ? 0.f : h * f.y);
    };
    for (int jj = tid; jj < N; jj += T) {
        if (!STEP) {
            irow[jj] = corrected(jj);
            if (jj <= N / 2) zhalf[jj] = zsplit[pix0 + N / 2 - jj];
            continue;
        }
        const float2 z = zsplit[pix0 + jj];
        if (keep_rows) {
            irow[jj] = corrected(jj);
            zrow[jj] = z;
        }
        float sn, cs;
        phase_tz(1.f, z, &sn, &cs);
        erow[jj] = make_float2(cs, -sn);
    }
    // Runtime plans whose last-stage butterflies take whole strips apart keep a mask per
    // strip of their first elements instead: one load for all of a butterfly's strips
    // (they span ntu strips in mask_span steps; at least 4, so the masks fit in occ's room).
    unsigned *mask = reinterpret_cast<unsigned *>(occ);
    const int last_L = F.L[F.nstages - (F.nstages > 2 && F.fuse[F.nstages - 2] ? 2 : 1)];
    const int mask_span = NP == 0 && last_L % TU == 0 && 4 * last_L <= Np ? last_L / TU : 0;
    int occ_tt = -1;
    const typename RowTwOf<NP>::type rt(tw, false, tid);        // the thread's twiddle bases, read once
    for (int p = p_begin; p < p_end; ++p) {
        const int pl = plane0 + p;
        const float t = (float)(pl + L.t_lo);
        float2 *plane = stack + (size_t)p * Np * Np;
        const int tt = pl / TT;
        __syncthreads();                     // row and z visible; the previous plane's last stage is done
        if (tt != occ_tt) {                  // uniform across the CTA
            const uint8_t *strips = col_occ + tt * L.ntu;
            if (mask_span > 0)
                for (int i = tid; i < mask_span; i += T) {
                    unsigned bits = 0u;
                    for (int m = 0; m * mask_span < L.ntu; ++m) bits |= (unsigned)(strips[i + m * mask_span] != 0) << m;
                    mask[i] = bits;
                }
            else
                for (int i = tid; i < L.ntu; i += T) occ[i] = strips[i];
            occ_tt = tt;
            __syncthreads();
        }
        // row x exp(-i phi), phi = 2 pi t z: (f.x cs + f.y sn, f.y cs - f.x sn), the products with f.x rounded first
        auto screened = [](float2 f, float sn, float cs) {
            return fma2(dup2(f.y), make_float2(sn, cs), mul2(dup2(f.x), make_float2(cs, -sn)));
        };
        if (!STEP) {
            for (int h = tid; h <= N / 2; h += T) {
                float sn, cs;
                phase_tz(t, zhalf[h], &sn, &cs);
                scr[h] = make_float2(cs, sn);
            }
            __syncthreads();
        } else if ((p - p_begin) % kScreenSteps == 0) {
            for (int jj = tid; jj < N; jj += T) {
                const float2 f = keep_rows ? irow[jj] : corrected(jj);
                float sn, cs;
                phase_tz(t, keep_rows ? zrow[jj] : zsplit[pix0 + jj], &sn, &cs);
                grow[jj] = screened(f, sn, cs);
            }
            __syncthreads();
        }
        const bool step = STEP && (p + 1 - p_begin) % kScreenSteps != 0 && p + 1 < p_end;   // uniform: advance g
        auto load = [&](auto pruned, int, int J0, int dJ, auto &v) {
            constexpr int R = length_of<decltype(v)>();
            constexpr bool P = decltype(pruned)::value;
            if constexpr (!STEP) {
                for_live<R, P>([&](int m) {
                    const unsigned jj = grid_to_crop(J0 + m * dJ, half, Np);
                    v[m] = make_float2(0.f, 0.f);
                    if (jj >= (unsigned)N) return;
                    const float2 s = scr[abs((int)jj - half)];
                    v[m] = screened(irow[jj], s.y, s.x);
                });
                return;
            } else if constexpr (NP == 0) {
                // (runtime plans: reading all steps first took more registers than it saved time)
                for_live<R, P>([&](int m) {
                    const unsigned jj = grid_to_crop(J0 + m * dJ, half, Np);
                    v[m] = make_float2(0.f, 0.f);
                    if (jj >= (unsigned)N) return;
                    v[m] = grow[jj];
                    if (step) grow[jj] = step_screen(v[m], erow[jj]);
                });
                return;
            }
            for_live<R, P>([&](int m) {
                const unsigned jj = grid_to_crop(J0 + m * dJ, half, Np);
                v[m] = jj < (unsigned)N ? grow[jj] : make_float2(0.f, 0.f);
            });
            if (!step) return;
            float2 e[R];
            for_live<R, P>([&](int m) {
                const unsigned jj = grid_to_crop(J0 + m * dJ, half, Np);
                if (jj < (unsigned)N) e[m] = erow[jj];
            });
            for_live<R, P>([&](int m) {
                const unsigned jj = grid_to_crop(J0 + m * dJ, half, Np);
                if (jj < (unsigned)N) grow[jj] = step_screen(v[m], e[m]);
            });
        };
        // columns of this plane's t-tile that no footprint touches are never read
        auto store = [&](auto, int, int R0, int dR, auto &v) {
            if (NP == 0 && mask_span > 0) {                      // one address and a stride
                float2 *at = plane + tiled_index(ii, R0, Np);
                const size_t stride = (size_t)(dR / CB) * Np * CB;
                const unsigned strips = mask[R0 / TU];
                for_live<length_of<decltype(v)>(), false>([&](int m) {
                    if (strips >> m & 1u) __stcs(at + m * stride, v[m]);
                });
                return;
            }
            for_live<length_of<decltype(v)>(), false>([&](int m) {
                const int R = R0 + m * dR;
                if (occ[R / TU]) __stcs(plane + tiled_index(ii, R, Np), v[m]);
            });
        };
        if constexpr (NP >= 512)
            fft_static_row<NP, row_threads_max<NP>(), CROP ? fftst::PRUNE_IN : 0>(sbuf, false, tid, load, store, rt);
        else
            fft_many<1, false>(sbuf, F, tw, tid, T, load, store);
    }
}

// A column CTA is short and waits for its columns' loads at DRAM latency.  In the
// forward direction, whose loads are the N rows of a block in one run, the CTA of
// a block's first column pair asks L2 for the rows of the block `ahead` CTAs later
// (about the CTAs resident at once; 0: it does not).  Worth it from N = 2048 on (366
// planes of N' = 4096: 10.98 -> 10.40 ms; N = 1024: 1.41 -> 1.43); inverse, where the
// loads are the occupied tiles, 512 bytes each, it cost more than it gave (10.96 -> 11.27).
constexpr int kAheadMinImage = 2048;
__device__ __forceinline__ void fetch_columns_ahead(const Launch &L, const uint8_t *__restrict__ col_occ, int plane0,
                                                    int ahead, const float2 *__restrict__ stack) {
    if (ahead == 0 || (blockIdx.x & 1) || threadIdx.x >= 4) return;      // a quarter of the rows each
    const unsigned x = blockIdx.x + (unsigned)ahead, pair = x % gridDim.x, plane = blockIdx.y + x / gridDim.x;
    if (plane >= gridDim.y || plane0 + (int)plane >= L.Nw) return;
    if (!col_occ[(plane0 + (int)plane) / TT * L.ntu + (int)pair * kPerCta / TU]) return;
    const unsigned bytes = (unsigned)(L.N / 4 * CB * sizeof(float2));
    const char *block = reinterpret_cast<const char *>(stack + (size_t)plane * L.Np * L.Np +
                                                       (size_t)(pair * kPerCta / CB) * L.Np * CB);
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                     __cvta_generic_to_global(block + (size_t)threadIdx.x * bytes)),
                 "r"(bytes)
                 : "memory");
}

template <int NP, bool CROP>
__global__ void __launch_bounds__(col_threads_max<NP>(), col_ctas<NP>())
fwd_cols_kernel(Launch L, FftPlan F, const float2 *__restrict__ tw, const uint8_t *__restrict__ tile_occ,
                const uint8_t *__restrict__ col_occ, int plane0, int ahead, float2 *__restrict__ stack) {
    extern __shared__ __align__(16) float2 sbuf[];
    const int Np = L.Np, half = L.N / 2;
    fetch_columns_ahead(L, col_occ, plane0, ahead, stack);
    const int R0 = blockIdx.x * kPerCta;                  // two of the four columns of a block
    const int tt = (plane0 + (int)blockIdx.y) / TT, tu = R0 / TU;
    if (plane0 + (int)blockIdx.y >= L.Nw) return;         // padding planes of the last t-tile: never read
    if (!col_occ[tt * L.ntu + tu]) return;                // no visibility reads these columns of this plane
    float2 *blk = stack + (size_t)blockIdx.y * Np * Np + (size_t)(R0 >> 2) * Np * CB + (R0 & 3);
    uint8_t *occ = reinterpret_cast<uint8_t *>(sbuf + kPerCta * (NP == 4096 ? fftst::kStride64 : F.stride));
    for (int i = threadIdx.x; i < L.ntv; i += blockDim.x) occ[i] = tile_occ[((size_t)tt * L.ntv + i) * L.ntu + tu];
    __syncthreads();
    // rows 0..N-1 hold the N transformed image rows; every other row is zero padding
    auto load = [&](auto pruned, int b, int S0, int dS, auto &v) {
        for_live<length_of<decltype(v)>(), decltype(pruned)::value>([&](int m) {
            const unsigned c = grid_to_crop(S0 + m * dS, half, Np);
            v[m] = c < 2u * half ? __ldcs(blk + (size_t)c * CB + b) : make_float2(0.f, 0.f);
        });
    };
    auto store = [&](auto, int b, int S0, int dS, auto &v) {
        for_live<length_of<decltype(v)>(), false>([&](int m) {
            const int S = S0 + m * dS;
            if (occ[S >> L.tv_log]) blk[(size_t)S * CB + b] = v[m];     // only tiles the gather reads
        });
    };
    column_fft<NP, false, CROP ? fftst::PRUNE_IN : 0>(sbuf, F, tw, load, store);
}

// -- gridding ----------------------------------------------------------------

template <int NP, bool CROP>
__global__ void __launch_bounds__(col_threads_max<NP>(), col_ctas<NP>())
inv_cols_kernel(Launch L, FftPlan F, const float2 *__restrict__ tw, const uint8_t *__restrict__ tile_occ,
                const uint8_t *__restrict__ col_occ, int plane0, float2 *__restrict__ stack) {
    extern __shared__ __align__(16) float2 sbuf[];
    const int Np = L.Np, half = L.N / 2;
    const int R0 = blockIdx.x * kPerCta;
    const int tt = (plane0 + (int)blockIdx.y) / TT, tu = R0 / TU;
    if (plane0 + (int)blockIdx.y >= L.Nw) return;         // padding planes of the last t-tile: inv_rows skips them
    if (!col_occ[tt * L.ntu + tu]) return;                // all-zero columns: inv_rows skips them too
    float2 *blk = stack + (size_t)blockIdx.y * Np * Np + (size_t)(R0 >> 2) * Np * CB + (R0 & 3);
    uint8_t *occ = reinterpret_cast<uint8_t *>(sbuf + kPerCta * (NP == 4096 ? fftst::kStride64 : F.stride));
    for (int i = threadIdx.x; i < L.ntv; i += blockDim.x) occ[i] = tile_occ[((size_t)tt * L.ntv + i) * L.ntu + tu];
    __syncthreads();
    // gridding wrote only occupied tiles; every other cell is zero
    auto load = [&](auto, int b, int S0, int dS, auto &v) {
        for_live<length_of<decltype(v)>(), false>([&](int m) {
            const int S = S0 + m * dS;
            v[m] = occ[S >> L.tv_log] ? __ldcs(blk + (size_t)S * CB + b) : make_float2(0.f, 0.f);
        });
    };
    // keep the N crop rows, compacted into rows 0..N-1 (all reads precede these writes)
    auto store = [&](auto pruned, int b, int S0, int dS, auto &v) {
        for_live<length_of<decltype(v)>(), decltype(pruned)::value>([&](int m) {
            const unsigned c = grid_to_crop(S0 + m * dS, half, Np);
            if (c < 2u * half) blk[(size_t)c * CB + b] = v[m];
        });
    };
    column_fft<NP, true, CROP ? fftst::PRUNE_OUT : 0>(sbuf, F, tw, load, store);
}

// -- TMA row copies and mbarriers ----------------------------------------------

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Wait for the phase of the given parity to complete, giving up after
// `polls` polls (kWaitPolls: a few hundred milliseconds): false if it did not
// complete.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, int polls = kWaitPolls) {
    for (int i = 0; i < polls; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        __nanosleep(64);
    }
    return false;
}
// Box of an image row: {8 floats, 1 row, box_blocks column blocks, 1 plane} of the stack's row map.
__device__ __forceinline__ void tma_row_box(float2 *dst, const CUtensorMap *map, int row, int block, int plane,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(block), "r"(plane), "r"(smem_addr(bar))
        : "memory");
}

// Shared memory of inv_rows: one or two 128-byte aligned row buffers (TMA
// destinations), the compensated sums, the half rows of z and screen (where they fit), two mbarriers and a flag.
struct RowsSmem {
    int buffers;          // 2: the next plane's row is copied while this one is transformed
    int half;             // 1: half rows of z and of the screen; 0: z from global memory
    size_t buf, bytes;
};
inline RowsSmem rows_smem(const FftPlan &F, int N) {
    const size_t buf = ((size_t)F.stride * sizeof(float2) + 127) / 128 * 128;
    auto layout = [&](int buffers, int half) {
        return RowsSmem{buffers, half, buf,
                        128 + buffers * buf + (size_t)N * sizeof(float4) + (half ? (N + 2) * sizeof(float2) : 0) + 32};
    };
    // As many CTAs per SM as registers allow come first: they cover each other's
    // barriers and waits.  For that the second buffer goes, if the last stage's inputs
    // fit in registers (dit_last_held), and then the half rows.
    const int last = F.nstages - 1;
    const bool held = compile_time_size(F.n) || F.nb[last] <= F.row_threads * (32 / F.radix[last]);
    for (int ctas = row_cta_limit(F); ctas > 1; --ctas) {
        for (const RowsSmem &r : {layout(2, 1), layout(1, 1), layout(2, 0), layout(1, 0)})
            if ((held || r.buffers == 2) && r.bytes <= cta_smem(ctas)) return r;
    }
    return layout(2, 1).bytes <= cta_smem(1) ? layout(2, 1) : layout(2, 0);
}

// HALF: shared memory keeps half a row of z and of the plane's screen exp(2 pi i t
// z).  z depends on l^2, so a pixel and its mirror image share both: the N/2 + 1
// screens are evaluated together as the plane begins, half the evaluations of one
// per output (which were a quarter of the kernel's instructions), in the room that
// a whole row of z took.  (Stepping the screen from plane to plane as fwd_rows does is
// cheaper still, but raised the error against the exact DFT from 2.7e-7 to 3.0e-7.)
//
// One CTA owns image row ii and an equal share of the chunk's planes (share
// blockIdx.y of gridDim.y): it sums them into a compensated accumulator in
// shared memory; the last FFT stage screens and accumulates.  Where a row is
// shared, every share keeps its own sums in acc (N x N per share), and the CTA
// that finishes the row last adds them up in share order, so the result does not
// depend on which one that is.  With share_planes > 0 (deterministic plans) share g
// owns planes [g share_planes, (g + 1) share_planes) of the plan instead, in
// whichever chunks they come, so that the sums do not depend on the chunks either.
//
// The rows come by TMA in boxes of up to 256 column blocks (8 KB), all
// completing on the buffer's mbarrier: with two buffers, plane p + 1's row is
// copied while plane p is transformed; with one (ONE_BUFFER) it is copied while
// the last stage, whose inputs are in registers by then, finishes plane p.  Strips no footprint touched hold stale
// data; the first FFT stage masks them to zero.  Every wait is bounded; a CTA
// that gives up waits (bounded) for the copy in flight and ends; *timeouts
// counts the rows left incomplete, once each however many shares and chunks
// gave up, and they are not written.
constexpr unsigned kRowIncomplete = 0x10000u;      // above the count of a row's finished shares
template <int NP, bool CROP, bool ONE_BUFFER, bool HALF>
__global__ void __launch_bounds__(row_threads_max<NP>(), row_ctas<NP>())
inv_rows_kernel(Launch L, FftPlan F, const float2 *__restrict__ tw, const __grid_constant__ CUtensorMap row_map,
                const uint8_t *__restrict__ col_occ, int plane0, int planes, int share_planes, int buf_slots,
                const float2 *__restrict__ zsplit, const float *__restrict__ corr, float4 *__restrict__ acc,
                unsigned *__restrict__ rows_done, int first, int last, float2 *__restrict__ dirty,
                unsigned long long *__restrict__ timeouts, int wait_polls) {
    extern __shared__ __align__(16) float2 sbuf[];
    constexpr int buffers = ONE_BUFFER ? 1 : 2;
    const int Np = L.Np, N = L.N, half = N / 2;
    const int ii = blockIdx.x, tid = threadIdx.x, T = NP ? row_threads_max<NP>() : (int)blockDim.x;
    const int R0 = NP ? fftst::Radices<NP ? NP : 512>::r0 : F.radix[0], nb = NP ? NP / 16 : F.nb[0];
    const int shares = gridDim.y, nvalid = min(planes, L.Nw - plane0);
    const int per = share_planes > 0 ? share_planes : (nvalid + shares - 1) / shares;
    const int own = (int)blockIdx.y * per - (share_planes > 0 ? plane0 : 0);
    const int p_begin = min(nvalid, max(0, own)), p_end = min(nvalid, max(0, own + per));
    if (p_begin == p_end && !first && !last) return;         // nothing to add in this chunk
    const size_t pix0 = (size_t)ii * N, image = (size_t)N * N;
    float4 *own_acc = acc + blockIdx.y * image;
    // 128-byte aligned start, by pointer arithmetic on sbuf so that every
    // access below stays a shared-memory access
    float2 *base = sbuf + ((128u - (smem_addr(sbuf) & 127u)) & 127u) / sizeof(float2);
    auto row_buf = [&](int k) { return base + (k & (buffers - 1)) * buf_slots; };
    float4 *srow = reinterpret_cast<float4 *>(base + buffers * buf_slots);   // N: (sum re, sum im, comp re, comp im)
    float2 *scr = reinterpret_cast<float2 *>(srow + N);                      // N/2 + 1 if HALF: exp(2 pi i t z)
    float2 *zhalf = scr + N / 2 + 1;                                         // N/2 + 1 if HALF: z
    uint64_t *bar = reinterpret_cast<uint64_t *>(scr + (HALF ? N + 2 : 0));  // 2
    volatile int &finisher = *reinterpret_cast<int *>(bar + 2);              // shared by the CTA
    const int warp = tid >> 5, lane = tid & 31;
    // warp 0: copy row ii of the share's k-th plane into buffer k mod buffers
    auto issue = [&](int k) {
        fence_proxy_async();                 // the buffer's last generic reads precede these writes
        uint64_t *b = &bar[k & (buffers - 1)];
        if (lane == 0) mbar_arrive_expect_tx(b, (unsigned)(Np * sizeof(float2)));
        __syncwarp();
        if (lane < F.boxes)
            tma_row_box(row_buf(k) + lane * F.box_blocks * CB, &row_map, ii, lane * F.box_blocks, p_begin + k, b);
    };
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_init_fence();
    }
    if (HALF)
        for (int h = tid; h <= N / 2; h += T) zhalf[h] = zsplit[pix0 + N / 2 - h];
    for (int jj = tid; jj < N; jj += T) {
        srow[jj] = first ? make_float4(0.f, 0.f, 0.f, 0.f) : own_acc[pix0 + jj];
    }
    const typename RowTwOf<NP>::type rt(tw, true, tid);
    __syncthreads();
    const int count = p_end - p_begin;
    if (warp == 0 && count > 0) issue(0);
    uint32_t live = 0;                       // strips of this thread's first-stage inputs, one t-tile
    int live_tt = -1;
    bool gave_up = false;                    // uniform
    for (int k = 0; k < count; ++k) {
        const int pl = plane0 + p_begin + k;
        const float t = (float)(pl + L.t_lo);
        const int tt = pl / TT;
        if (tt != live_tt) {                 // threads past nb own no first-stage butterfly
            live = 0;
            if (tid < nb) {
#pragma unroll 4
                for (int m = 0; m < R0; ++m)
                    live |= (uint32_t)(__ldg(col_occ + tt * L.ntu + (m * nb + tid) / TU) != 0) << m;
            }
            live_tt = tt;
        }
        uint64_t *b = &bar[k & (buffers - 1)];
        const unsigned parity = (buffers == 2 ? k >> 1 : k) & 1;
        const bool ok = mbar_wait(b, parity, wait_polls);
        if (__syncthreads_or(!ok)) {         // uniform: give up on this row
            if (tid == 0) mbar_wait(b, parity);              // drain the copy in flight (full limit)
            gave_up = true;
            break;
        }
        // every thread is past plane k - 1, so its buffer is free for plane k + 1
        if (warp == 0 && buffers == 2 && k + 1 < count) issue(k + 1);
        // the screen of this plane, read by the last stage (the stages' barriers lie between)
        if (HALF)
            for (int h = tid; h <= N / 2; h += T) {
                float sn, cs;
                phase_tz(t, zhalf[h], &sn, &cs);
                scr[h] = make_float2(cs, sn);
            }
        // a few outputs at a time: their screens and sums are read before any sum is written
        auto store = [&](auto pruned, int, int J0, int dJ, auto &v) {
            constexpr int R = length_of<decltype(v)>(), G = NP == 0 && ONE_BUFFER ? 2 : 4;
            constexpr bool P = decltype(pruned)::value;
#pragma unroll
            for (int m0 = 0; m0 < R; m0 += G) {
                if (P && m0 >= R / 4 && m0 + G <= 3 * R / 4) continue;
                // (runtime plans: keep the compiler from reading every group's z and sums first)
                if (NP == 0) asm volatile("" ::: "memory");
                float2 z[G];
                float4 a[G];
                unsigned at[G];                                  // outputs outside the crop read the row's last pixel
                auto wanted = [&](int i) { return m0 + i < R && !(P && m0 + i >= R / 4 && m0 + i < 3 * R / 4); };
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    if (!wanted(i)) continue;
                    at[i] = grid_to_crop(J0 + (m0 + i) * dJ, half, Np);
                    const int jj = (int)min(at[i], (unsigned)N - 1u);
                    z[i] = HALF ? scr[abs(jj - half)] : __ldg(zsplit + pix0 + jj);
                    a[i] = srow[jj];
                }
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    if (!wanted(i) || at[i] >= (unsigned)N) continue;
                    float sn = z[i].y, cs = z[i].x;
                    if (!HALF) phase_tz(t, z[i], &sn, &cs);
                    float2 sum = make_float2(a[i].x, a[i].y), comp = make_float2(a[i].z, a[i].w);
                    kahan_add(sum, comp, cmul_rot(v[m0 + i], make_float2(cs, sn), make_float2(-sn, cs)));
                    srow[at[i]] = make_float4(sum.x, sum.y, comp.x, comp.y);
                }
            }
        };
        auto between = [&] {
            if (warp == 0 && k + 1 < count) issue(k + 1);
        };
        if constexpr (NP >= 512)
            fft_static_inplace<NP, row_threads_max<NP>(), ONE_BUFFER, CROP ? fftst::PRUNE_OUT : 0>(
                row_buf(k), true, tid, between, store, rt, live);
        else
            fft_inplace<ONE_BUFFER>(row_buf(k), F, tw, tid, T, between, store, live);
    }
    __syncthreads();
    // a row that misses a plane of any chunk is marked in its counter
    if (gave_up && tid == 0) atomicOr(&rows_done[ii], kRowIncomplete);
    if (!gave_up && !(last && shares == 1))
        for (int jj = tid; jj < N; jj += T) own_acc[pix0 + jj] = srow[jj];
    if (!last) return;
    // the counter's low bits hold the finished shares; the last one to finish leaves it
    // zero for the next call, counts an incomplete row once and does not write it
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const unsigned all = atomicAdd(&rows_done[ii], 1u) + 1u;
        finisher = (all & (kRowIncomplete - 1u)) == (unsigned)shares ? 1 : 0;
        if (finisher) {
            rows_done[ii] = 0u;
            if (all & kRowIncomplete) {
                atomicAdd(timeouts, 1ull);
                finisher = 0;
            }
        }
        __threadfence();
    }
    __syncthreads();
    if (!finisher) return;
    for (int jj = tid; jj < N; jj += T) {
        float4 a = shares == 1 ? srow[jj] : __ldcg(acc + pix0 + jj);
        float2 sum = make_float2(a.x, a.y), comp = make_float2(a.z, a.w);
        for (int g = 1; g < shares; ++g) {
            a = __ldcg(acc + g * image + pix0 + jj);
            add_sums(sum, comp, a);
        }
        const float h = corr[pix0 + jj];
        dirty[pix0 + jj] = make_float2(h * (sum.x - comp.x), L.fold ? 0.f : h * (sum.y - comp.y));
    }
}

// transform buffers + one occupancy byte per strip (at most N'/16 or N'/32 of them)
inline size_t smem2(const FftPlan &F) {
    const int slots = F.n == 4096 ? std::max(F.stride, fftst::kStride64) : F.stride;
    return (size_t)kPerCta * slots * sizeof(float2) + F.n / TU + 16;
}
inline size_t smem_fwd_rows(const FftPlan &F, int N, bool keep_rows) {
    return (size_t)F.stride * sizeof(float2) + (size_t)N * (keep_rows ? 4 : 2) * sizeof(float2) + F.n / TU + 32;
}
// fwd_rows steps its screen where four rows leave room for two CTAs per SM: N up to
// about 2400 at x0 = 1/4.  Larger sizes evaluate it on every plane (the reason: at the kernel).
inline bool fwd_rows_step(const FftPlan &F, int N) { return smem_fwd_rows(F, N, true) <= cta_smem(2); }
// a stepping fwd_rows keeps the image row and z in shared memory where that costs no resident CTA
inline bool fwd_rows_keep(const FftPlan &F, int N) {
    auto fit = [&](bool keep) {
        return std::min<size_t>(row_cta_limit(F), 228 * 1024 / (smem_fwd_rows(F, N, keep) + 1024));
    };
    return fwd_rows_step(F, N) && fit(true) == fit(false);
}
// CTAs per image row in fwd_rows (each takes an equal share of the planes):
// enough rows x groups for about 32 CTAs per SM over the launch,
// so the SMs that finish first in the last round idle for a short CTA, not a long one
inline int row_groups(int N, int planes, int sms) {
    const int want = (32 * sms + N - 1) / N;
    return want < 1 ? 1 : (want > planes ? (planes > 0 ? planes : 1) : want);
}
// Raise a kernel's dynamic shared-memory limit to the device's opt-in maximum
// (after checking that this plan's need fits): kernels are shared by every
// plan, so a limit set to one plan's need could be too low for another's.
template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (bytes > (size_t)optin) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
}

// The stack as a 4-D FP32 tensor for TMA row copies: {8 floats of a column
// block's row, N' rows, N'/4 blocks, P planes}, boxes of box_blocks (FftPlan) blocks of one row.
cudaError_t row_tensor_map(const ws_plan_s *p, CUtensorMap *map);

// Launchers of one FFT variant.
template <int NP>
struct Transforms {
    // N <= N' <= 2048 fits four rows in half an SM's shared memory, and so does N = N'/2 = 2048
    static constexpr bool kMayNotStep = NP == 0 || NP == 4096;
    static cudaError_t setup(const FftPlan &F, const FftPlan &inv, int N) {
        cudaError_t e;
        const size_t rows = smem_fwd_rows(F, N, fwd_rows_keep(F, N));
        if ((e = allow_smem(fwd_rows_kernel<NP, false, true>, rows)) != cudaSuccess) return e;
        if constexpr (NP != 0)
            if ((e = allow_smem(fwd_rows_kernel<NP, true, true>, rows)) != cudaSuccess) return e;
        if constexpr (kMayNotStep)
            if ((e = allow_smem(fwd_rows_kernel<NP, false, false>, rows)) != cudaSuccess) return e;
        if ((e = allow_smem(fwd_cols_kernel<NP, false>, smem2(F))) != cudaSuccess) return e;
        if constexpr (NP != 0)
            if ((e = allow_smem(fwd_cols_kernel<NP, true>, smem2(F))) != cudaSuccess) return e;
        if ((e = allow_smem(inv_cols_kernel<NP, false>, smem2(inv))) != cudaSuccess) return e;
        if constexpr (NP != 0)
            if ((e = allow_smem(inv_cols_kernel<NP, true>, smem2(inv))) != cudaSuccess) return e;
        const size_t inv_rows = rows_smem(inv, N).bytes;
        auto allow = [&](auto crop) {
            constexpr bool C = decltype(crop)::value;
            cudaError_t r = allow_smem(inv_rows_kernel<NP, C, false, true>, inv_rows);
            if (r == cudaSuccess) r = allow_smem(inv_rows_kernel<NP, C, false, false>, inv_rows);
            if (r == cudaSuccess) r = allow_smem(inv_rows_kernel<NP, C, true, true>, inv_rows);
            return r == cudaSuccess ? allow_smem(inv_rows_kernel<NP, C, true, false>, inv_rows) : r;
        };
        e = allow(std::false_type{});
        if constexpr (NP != 0)
            if (e == cudaSuccess) e = allow(std::true_type{});
        return e;
    }
    // Runs go(std::bool_constant): whether the crop is the centred half (compile-time plans only).
    template <class Go>
    static void with_crop(const Launch &L, Go go) {
        if constexpr (NP != 0) {
            if (crop_half<NP>(L)) {
                go(std::true_type{});
                return;
            }
        }
        go(std::false_type{});
    }
    // column CTAs resident on the GPU, a multiple of the two of a block
    static int columns_ahead(const FftPlan &F, int sms) {
        const int by_smem = (int)(228 * 1024 / (smem2(F) + 1024));
        const int by_regs = col_ctas<NP>() * col_threads_max<NP>() / col_threads(F);
        return std::max(1, std::min(by_smem, by_regs)) * sms / 2 * 2;
    }
    static int row_threads(const FftPlan &F) { return NP ? row_threads_max<NP>() : F.row_threads; }
    static int col_threads(const FftPlan &F) { return NP ? col_threads_max<NP>() : F.col_threads; }
    static cudaError_t fwd_rows(const ws_plan_s *p, const float2 *image, int chunk, int planes, cudaStream_t s) {
        const bool keep = fwd_rows_keep(p->fft_fwd, p->L.N);
        const dim3 grid(p->L.N, row_groups(p->L.N, planes, p->sms));
        auto go = [&](auto kernel) {
            kernel<<<grid, row_threads(p->fft_fwd), smem_fwd_rows(p->fft_fwd, p->L.N, keep), s>>>(
                p->L, p->fft_fwd, p->d_tw, image, p->d_corr, p->d_zsplit, p->d_col_occ, chunk * p->P, planes,
                keep ? 1 : 0, p->d_stack);
        };
        if (!fwd_rows_step(p->fft_fwd, p->L.N)) {
            if constexpr (kMayNotStep)
                go(fwd_rows_kernel<NP, false, false>);
            else
                return cudaErrorInvalidValue;
            return cudaGetLastError();
        }
        with_crop(p->L, [&](auto crop) { go(fwd_rows_kernel<NP, decltype(crop)::value, true>); });
        return cudaGetLastError();
    }
    static cudaError_t fwd_cols(const ws_plan_s *p, int chunk, int planes, cudaStream_t s) {
        const dim3 grid(p->L.Np / kPerCta, planes);
        with_crop(p->L, [&](auto crop) {
            fwd_cols_kernel<NP, decltype(crop)::value><<<grid, col_threads(p->fft_fwd), smem2(p->fft_fwd), s>>>(
                p->L, p->fft_fwd, p->d_tw, p->d_tile_occ, p->d_col_occ, chunk * p->P,
                p->L.N >= kAheadMinImage ? columns_ahead(p->fft_fwd, p->sms) : 0, p->d_stack);
        });
        return cudaGetLastError();
    }
    static cudaError_t inv_cols(const ws_plan_s *p, int chunk, int planes, cudaStream_t s) {
        const dim3 grid(p->L.Np / kPerCta, planes);
        with_crop(p->L, [&](auto crop) {
            inv_cols_kernel<NP, decltype(crop)::value><<<grid, col_threads(p->fft_inv), smem2(p->fft_inv), s>>>(
                p->L, p->fft_inv, p->d_tw, p->d_tile_occ, p->d_col_occ, chunk * p->P, p->d_stack);
        });
        return cudaGetLastError();
    }
    static cudaError_t inv_rows(const ws_plan_s *p, int chunk, int planes, bool first, bool last, float2 *dirty,
                                cudaStream_t s) {
        CUtensorMap map{};
        const cudaError_t e = row_tensor_map(p, &map);
        if (e != cudaSuccess) return e;
        const RowsSmem sm = rows_smem(p->fft_inv, p->L.N);
        auto go = [&](auto kernel) {
            kernel<<<dim3(p->L.N, p->row_shares), row_threads(p->fft_inv), sm.bytes, s>>>(
                p->L, p->fft_inv, p->d_tw, map, p->d_col_occ, chunk * p->P, planes, p->share_planes,
                (int)(sm.buf / sizeof(float2)), p->d_zsplit, p->d_corr, p->d_acc, p->d_rows_done, first ? 1 : 0,
                last ? 1 : 0, dirty, p->d_drop + 2, p->wait_polls);
        };
        with_crop(p->L, [&](auto crop) {
            constexpr bool C = decltype(crop)::value;
            if (sm.buffers == 1)
                sm.half ? go(inv_rows_kernel<NP, C, true, true>) : go(inv_rows_kernel<NP, C, true, false>);
            else
                sm.half ? go(inv_rows_kernel<NP, C, false, true>) : go(inv_rows_kernel<NP, C, false, false>);
        });
        return cudaGetLastError();
    }
};

// Entry points of one variant, exported by the translation unit that
// instantiates it (so every kernel is compiled exactly once).
struct Ops {
    cudaError_t (*setup)(const FftPlan &, const FftPlan &, int);
    cudaError_t (*fwd_rows)(const ws_plan_s *, const float2 *, int, int, cudaStream_t);
    cudaError_t (*fwd_cols)(const ws_plan_s *, int, int, cudaStream_t);
    cudaError_t (*inv_cols)(const ws_plan_s *, int, int, cudaStream_t);
    cudaError_t (*inv_rows)(const ws_plan_s *, int, int, bool, bool, float2 *, cudaStream_t);
};

template <int NP>
constexpr Ops ops_of() {
    return Ops{&Transforms<NP>::setup, &Transforms<NP>::fwd_rows, &Transforms<NP>::fwd_cols,
               &Transforms<NP>::inv_cols, &Transforms<NP>::inv_rows};
}

const Ops &ops_runtime();
const Ops &ops_512();
const Ops &ops_1024();
const Ops &ops_2048();
const Ops &ops_4096();

}  // namespace tf
}  // namespace ws
