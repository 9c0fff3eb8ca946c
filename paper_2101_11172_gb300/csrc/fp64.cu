// FP64 path of gridding and degridding (plans made with WS_FLAG_FP64).
//
// The single-precision path is limited by FP32 rounding near 3e-7 relative,
// while the method's own bound E falls far lower for wider kernels (E of
// Eq. norm_bound is 6e-13 at W = 12 and reaches double-precision level at
// W = 14, x0 = 1/4; Section 6.3).  This path keeps everything in FP64 --
// coordinates, weights (the Chebyshev series of the plan's fit, evaluated
// by Clenshaw's recurrence), the w-stack, the plane transforms, the screens
// and the sums -- so that its error against the exact DFT follows sqrt(3) E
// down to W = 14.  It exists to measure the method's error, not for large
// problems: the w-planes are taken a chunk at a time (planes64, as many as fit in
// 2 GB and in the memory budget of a stack), Algorithm 5 and Algorithm 6 step by step, with FP64 atomics
// for the spread and a shared-memory FFT per line.
//
// Work split.  A warp takes a visibility through all of a chunk's planes: its 3W
// weights are evaluated once (one per lane; a Clenshaw chain of some thirty
// dependent steps) and its W^2 cells go to the lanes.  One thread per visibility
// and plane, with the weights evaluated anew for each plane, kept 4001 threads on
// 152 SMs busy for 64 and 81 us per plane (W = 12); this way the whole case of 29
// planes takes less than that.  The transforms take several lines per CTA and
// all planes of the chunk per launch, with the screens, crops and zero padding in
// their loads and stores.
//
// Layout: planes of N' x N' complex128, row S (v) by column R (u), both modulo
// N' as in the FP32 path; images N x N complex128; visibilities complex128.
#include <math.h>

#include <algorithm>

#include "ws_internal.hpp"

namespace ws {
namespace {

struct VisRec64 {
    int r0, s0, t0, folded;     // t0 < 0: dropped
    double nux, nuy, nuz;
    double pre_re, pre_im;      // exp(+2 pi i w (n0 - 1))
};

__device__ __forceinline__ int wrap_index64(double x, int n) {
    long long i = (long long)x;
    if (i < -n || i >= 2LL * n) i %= n;
    if (i < 0) i += n;
    if (i >= n) i -= n;
    return (int)i;
}

// c_i(nu) = sum_k cheb[i][k] T_k(2 nu) by Clenshaw's recurrence.
__device__ __forceinline__ double tap_weight(const double *__restrict__ cheb, int deg, int i, double nu) {
    const double *c = cheb + (size_t)i * (deg + 1);
    const double y = 2.0 * nu;
    double b1 = 0.0, b2 = 0.0;
    for (int k = deg; k >= 1; --k) {
        const double b0 = 2.0 * y * b1 - b2 + c[k];
        b2 = b1;
        b1 = b0;
    }
    return y * b1 - b2 + c[0];
}

__global__ void prep64_kernel(Launch L, const double *__restrict__ uvw, int64_t M, VisRec64 *__restrict__ rec,
                              unsigned long long *__restrict__ drop) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    double u = uvw[3 * k], v = uvw[3 * k + 1], w = uvw[3 * k + 2];
    const bool folded = L.fold && w < 0.0;     // Section 5.4: conjugate visibility at -(u, v, w)
    if (folded) {
        u = -u;
        v = -v;
        w = -w;
    }
    const int W = L.W;
    VisRec64 r{0, 0, -1, folded ? 1 : 0, 0.0, 0.0, 0.0, 1.0, 0.0};
    const double up = u * L.uv_scale, vp = v * L.uv_scale, wp = w * L.nscale;
    if (!(fabs(up) < 1e15) || !(fabs(vp) < 1e15)) {
        atomicAdd(&drop[0], 1ull);
        rec[k] = r;
        return;
    }
    const double ft = floor(wp + 0.5 * W);
    const double t0 = ft - (W - 1) - L.t_lo;
    if (!(t0 >= 0.0 && t0 + W <= (double)L.Nw)) {
        atomicAdd(&drop[1], 1ull);
        rec[k] = r;
        return;
    }
    const double fu = floor(up + 0.5 * W), fv = floor(vp + 0.5 * W);
    r.r0 = wrap_index64(fu - (W - 1), L.Np);
    r.s0 = wrap_index64(fv - (W - 1), L.Np);
    r.t0 = (int)t0;
    r.nux = up + 0.5 * (W - 1) - fu;
    r.nuy = vp + 0.5 * (W - 1) - fv;
    r.nuz = wp + 0.5 * (W - 1) - ft;
    double turns = w * L.n0m1;
    turns -= rint(turns);
    sincospi(2.0 * turns, &r.pre_im, &r.pre_re);
    rec[k] = r;
}

constexpr int kThreads64 = 128, kWarps64 = kThreads64 / 32;

// The chunk's part of a visibility: taps [c_lo, c_hi] along w; its 3W weights
// (u taps, v taps, w taps) go to w[], one per lane and round.  False if there is none.
__device__ __forceinline__ bool visibility_weights(const Launch &L, const double *__restrict__ cheb, int deg,
                                                   const VisRec64 &r, int p0, int planes, int lane, double *w,
                                                   int &c_lo, int &c_hi) {
    c_lo = max(0, p0 - r.t0);
    c_hi = min(L.W - 1, p0 + planes - 1 - r.t0);
    if (r.t0 < 0 || c_lo > c_hi) return false;           // uniform across the warp
    __syncwarp();                                        // the previous visibility's weights are read
    for (int l = lane; l < 3 * L.W; l += 32) {
        const int axis = l / L.W, i = l - axis * L.W;
        w[l] = tap_weight(cheb + (axis == 2 ? (size_t)L.W * (deg + 1) : 0), deg, i,
                          axis == 0 ? r.nux : (axis == 1 ? r.nuy : r.nuz));
    }
    __syncwarp();
    return true;
}

// Algorithm 5 steps 2-3a for planes p0 .. p0 + planes - 1: a warp adds
// V exp(2 pi i w (n0-1)) C_x C_y C_z to its visibility's cells.
__global__ void __launch_bounds__(kThreads64)
spread64_kernel(Launch L, const double *__restrict__ cheb, int deg, const VisRec64 *__restrict__ rec,
                const double2 *__restrict__ vis, int64_t M, int p0, int planes, double2 *__restrict__ stack) {
    __shared__ double weights[kWarps64][3 * kMaxW64];
    const int lane = threadIdx.x & 31, W = L.W, Np = L.Np;
    double *w = weights[threadIdx.x >> 5];
    const int64_t nwarps = (int64_t)gridDim.x * kWarps64;
    const size_t plane = (size_t)Np * Np;
    for (int64_t k = (int64_t)blockIdx.x * kWarps64 + (threadIdx.x >> 5); k < M; k += nwarps) {
        const VisRec64 r = rec[k];
        int c_lo, c_hi;
        if (!visibility_weights(L, cheb, deg, r, p0, planes, lane, w, c_lo, c_hi)) continue;
        double2 V = vis[k];
        if (r.folded) V.y = -V.y;
        const double vr = V.x * r.pre_re - V.y * r.pre_im, vi = V.x * r.pre_im + V.y * r.pre_re;
        for (int q = lane; q < W * W; q += 32) {
            const int b = q / W, a = q - b * W;
            const double wab = w[a] * w[W + b], xr = vr * wab, xi = vi * wab;
            double2 *cell =
                stack + (size_t)((r.s0 + b) % Np) * Np + (r.r0 + a) % Np + (size_t)(r.t0 + c_lo - p0) * plane;
            for (int c = c_lo; c <= c_hi; ++c, cell += plane) {
                const double wz = w[2 * W + c];
                atomicAdd(&cell->x, xr * wz);
                atomicAdd(&cell->y, xi * wz);
            }
        }
    }
}

// Algorithm 6 step 4 for planes p0 .. p0 + planes - 1: a warp adds
// sum F C_x C_y C_z over its visibility's cells to acc.
__global__ void __launch_bounds__(kThreads64)
gather64_kernel(Launch L, const double *__restrict__ cheb, int deg, const VisRec64 *__restrict__ rec, int64_t M, int p0,
                int planes, const double2 *__restrict__ stack, double2 *__restrict__ acc) {
    __shared__ double weights[kWarps64][3 * kMaxW64];
    const int lane = threadIdx.x & 31, W = L.W, Np = L.Np;
    double *w = weights[threadIdx.x >> 5];
    const int64_t nwarps = (int64_t)gridDim.x * kWarps64;
    const size_t plane = (size_t)Np * Np;
    for (int64_t k = (int64_t)blockIdx.x * kWarps64 + (threadIdx.x >> 5); k < M; k += nwarps) {
        const VisRec64 r = rec[k];
        int c_lo, c_hi;
        if (!visibility_weights(L, cheb, deg, r, p0, planes, lane, w, c_lo, c_hi)) continue;
        double sr = 0.0, si = 0.0;
        for (int q = lane; q < W * W; q += 32) {
            const int b = q / W, a = q - b * W;
            const double2 *cell =
                stack + (size_t)((r.s0 + b) % Np) * Np + (r.r0 + a) % Np + (size_t)(r.t0 + c_lo - p0) * plane;
            double cr = 0.0, ci = 0.0;
            for (int c = c_lo; c <= c_hi; ++c, cell += plane) {
                const double2 F = *cell;
                cr += w[2 * W + c] * F.x;
                ci += w[2 * W + c] * F.y;
            }
            const double wab = w[a] * w[W + b];
            sr += wab * cr;
            si += wab * ci;
        }
        for (int o = 16; o > 0; o >>= 1) {
            sr += __shfl_xor_sync(0xffffffffu, sr, o);
            si += __shfl_xor_sync(0xffffffffu, si, o);
        }
        if (lane == 0) acc[k] = make_double2(acc[k].x + sr, acc[k].y + si);
    }
}

// -- transforms ----------------------------------------------------------------
//
// A CTA transforms `lines` lines of n = 2^logn points in shared memory (n x
// lines at most kFftPoints64).  Points are loaded in bit-reversed order; a pass
// then does two radix-2 levels in registers, so log2(n) levels take half as many
// trips through shared memory.
constexpr int kFftPoints64 = 4096, kFftThreads64 = 256;
inline int fft_lines64(int n) { return std::max(1, std::min(16, kFftPoints64 / n)); }

__device__ __forceinline__ double2 cmul64(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ int rev64(int i, int logn) { return (int)(__brev((unsigned)i) >> (32 - logn)); }
__device__ __forceinline__ int crop64(int c, int half, int Np) { return c < half ? c - half + Np : c - half; }

__device__ __forceinline__ void fft64_shared(double2 *buf, int n, int logn, int lines, const double2 *__restrict__ tw,
                                             bool inverse) {
    int s = 0;
    __syncthreads();
    if (logn & 1) {
        for (int q = threadIdx.x; q < lines * n / 2; q += blockDim.x) {
            const double2 a = buf[2 * q], b = buf[2 * q + 1];
            buf[2 * q] = make_double2(a.x + b.x, a.y + b.y);
            buf[2 * q + 1] = make_double2(a.x - b.x, a.y - b.y);
        }
        s = 1;
        __syncthreads();
    }
    for (; s < logn; s += 2) {
        const int h = 1 << s;
        for (int q = threadIdx.x; q < lines * (n / 4); q += blockDim.x) {
            const int line = q / (n / 4), i = q - line * (n / 4), j = i & (h - 1);
            double2 *x = buf + line * n + ((i - j) << 2) + j;
            double2 w1 = tw[j << (logn - 1 - s)], w2 = tw[j << (logn - 2 - s)];   // level s, level s + 1
            if (inverse) {
                w1.y = -w1.y;
                w2.y = -w2.y;
            }
            const double2 a = x[0], b = cmul64(x[h], w1), c = x[2 * h], d = cmul64(x[3 * h], w1);
            const double2 a1 = make_double2(a.x + b.x, a.y + b.y), b1 = make_double2(a.x - b.x, a.y - b.y);
            const double2 c1 = cmul64(make_double2(c.x + d.x, c.y + d.y), w2);
            const double2 t = cmul64(make_double2(c.x - d.x, c.y - d.y), w2);
            // the other pair's twiddle is w2 times -i (forward) or +i (inverse)
            const double2 d1 = inverse ? make_double2(-t.y, t.x) : make_double2(t.y, -t.x);
            x[0] = make_double2(a1.x + c1.x, a1.y + c1.y);
            x[2 * h] = make_double2(a1.x - c1.x, a1.y - c1.y);
            x[h] = make_double2(b1.x + d1.x, b1.y + d1.y);
            x[3 * h] = make_double2(b1.x - d1.x, b1.y - d1.y);
        }
        __syncthreads();
    }
}

// exp(2 pi i t z), argument reduced in FP64
__device__ __forceinline__ double2 screen64(double t, double z) {
    double tz = t * z, s, c;
    tz -= rint(tz);
    sincospi(2.0 * tz, &s, &c);
    return make_double2(c, s);
}

// Algorithm 6 steps 2-3c, first half: image rows x correction x exp(-2 pi i t z), zero pad, DFT along u.
__global__ void __launch_bounds__(kFftThreads64)
fwd_rows64_kernel(Launch L, int logn, int lines, const double2 *__restrict__ tw, const double *__restrict__ corr,
                  const double2 *__restrict__ image, const double *__restrict__ z, int p0, double2 *__restrict__ stack) {
    extern __shared__ double2 buf64[];
    const int n = L.Np, N = L.N, half = N / 2, row0 = blockIdx.x * lines;
    const double t = (double)(p0 + (int)blockIdx.y + L.t_lo);
    double2 *plane = stack + (size_t)blockIdx.y * n * n;
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) {
        const int l = q >> logn, g = q & (n - 1), row = row0 + l;
        double2 v = make_double2(0.0, 0.0);
        if (row < N && (g < half || g >= n - half)) {
            const size_t i = (size_t)row * N + (g < half ? g + half : g - (n - half));
            const double2 f = image[i], e = screen64(t, z[i]);
            const double fr = corr[i] * f.x, fi = L.fold ? 0.0 : corr[i] * f.y;
            v = make_double2(fr * e.x + fi * e.y, fi * e.x - fr * e.y);
        }
        buf64[l * n + rev64(g, logn)] = v;
    }
    fft64_shared(buf64, n, logn, lines, tw, false);
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) {
        const int l = q >> logn, g = q & (n - 1), row = row0 + l;
        if (row < N) plane[(size_t)crop64(row, half, n) * n + g] = buf64[q];
    }
}

// DFT along v of `lines` columns: forward, from the N crop rows (the others are
// zero padding) to all rows; inverse, from all rows to the crop rows.
__global__ void __launch_bounds__(kFftThreads64)
cols64_kernel(Launch L, int logn, int lines, const double2 *__restrict__ tw, int inverse, double2 *__restrict__ stack) {
    extern __shared__ double2 buf64[];
    const int n = L.Np, half = L.N / 2;
    double2 *col = stack + (size_t)blockIdx.y * n * n + blockIdx.x * lines;
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) {
        const int i = q / lines, l = q - i * lines;
        const bool live = inverse || i < half || i >= n - half;
        buf64[l * n + rev64(i, logn)] = live ? col[(size_t)i * n + l] : make_double2(0.0, 0.0);
    }
    fft64_shared(buf64, n, logn, lines, tw, inverse != 0);
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) {
        const int i = q / lines, l = q - i * lines;
        if (!inverse || i < half || i >= n - half) col[(size_t)i * n + l] = buf64[l * n + i];
    }
}

// Algorithm 5 steps 3b-4, second half: DFT along u of the crop rows, crop
// columns x exp(+2 pi i t z), left in the first N cells of each crop row.
__global__ void __launch_bounds__(kFftThreads64)
inv_rows64_kernel(Launch L, int logn, int lines, const double2 *__restrict__ tw, const double *__restrict__ z, int p0,
                  double2 *__restrict__ stack) {
    extern __shared__ double2 buf64[];
    const int n = L.Np, N = L.N, half = N / 2, row0 = blockIdx.x * lines;
    const double t = (double)(p0 + (int)blockIdx.y + L.t_lo);
    double2 *plane = stack + (size_t)blockIdx.y * n * n;
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) {
        const int l = q >> logn, g = q & (n - 1), row = row0 + l;
        buf64[l * n + rev64(g, logn)] =
            row < N ? plane[(size_t)crop64(row, half, n) * n + g] : make_double2(0.0, 0.0);
    }
    fft64_shared(buf64, n, logn, lines, tw, true);
    for (int q = threadIdx.x; q < lines * N; q += blockDim.x) {
        const int l = q / N, j = q - l * N, row = row0 + l;
        if (row >= N) break;
        plane[(size_t)crop64(row, half, n) * n + j] =
            cmul64(buf64[l * n + crop64(j, half, n)], screen64(t, z[(size_t)row * N + j]));
    }
}

// Algorithm 5 steps 4-5: the sum over the chunk's planes, and after the last chunk dirty =
// h_x h_y h_z D (real part only for a folded real-sky plan).
__global__ void sum_planes64_kernel(Launch L, const double *__restrict__ corr, const double2 *__restrict__ stack,
                                    int planes, int first, int last, double2 *__restrict__ acc,
                                    double2 *__restrict__ dirty) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int N = L.N, n = L.Np;
    if (i >= (int64_t)N * N) return;
    const int row = (int)(i / N), col = (int)(i % N);
    const double2 *p = stack + (size_t)crop64(row, N / 2, n) * n + col;
    double2 a = first ? make_double2(0.0, 0.0) : acc[i];
    for (int k = 0; k < planes; ++k, p += (size_t)n * n) {
        a.x += p->x;
        a.y += p->y;
    }
    if (last)
        dirty[i] = make_double2(corr[i] * a.x, L.fold ? 0.0 : corr[i] * a.y);
    else
        acc[i] = a;
}

// Algorithm 6 step 5: x exp(-2 pi i w (n0 - 1)); folded visibilities conjugated.
__global__ void finish_degrid64_kernel(const VisRec64 *__restrict__ rec, int64_t M, double2 *__restrict__ vis) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    const VisRec64 r = rec[k];
    if (r.t0 < 0) {
        vis[k] = make_double2(0.0, 0.0);
        return;
    }
    const double2 a = vis[k];
    double2 out = make_double2(a.x * r.pre_re + a.y * r.pre_im, a.y * r.pre_re - a.x * r.pre_im);
    if (r.folded) out.y = -out.y;
    vis[k] = out;
}

inline unsigned blocks64(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Warps of a resident grid for M visibilities.
inline unsigned vis_blocks64(const ws_plan_s *p, int64_t M) {
    return (unsigned)std::min<int64_t>((M + kWarps64 - 1) / kWarps64, (int64_t)p->sms * 16);
}

// Launch shapes of the transforms of `planes` planes.
struct Fft64Launch {
    int lines;
    size_t smem;
    dim3 rows, cols;
    Fft64Launch(const Launch &L, int planes)
        : lines(fft_lines64(L.Np)), smem((size_t)lines * L.Np * sizeof(double2)),
          rows((L.N + lines - 1) / lines, planes), cols(L.Np / lines, planes) {}
};

}  // namespace

size_t fp64_record_bytes() { return sizeof(VisRec64); }

// Planes per chunk: as many as fit in 2 GB and in `budget` bytes, at least one.
int fp64_planes(int Np, int Nw, size_t budget) {
    constexpr size_t kPlaneBytes64 = (size_t)2 << 30;
    const size_t fit = std::min(kPlaneBytes64, budget) / ((size_t)Np * Np * sizeof(double2));
    return (int)std::max<size_t>(1, std::min<size_t>(fit, (size_t)Nw));
}

// The limit belongs to the kernel and every plan on the device shares it, so it is raised to what the
// largest line count needs (64 KB) whatever this plan's size: a limit set to one plan's need would
// make the launches of a larger one fail.
cudaError_t fp64_setup() {
    const int smem = (int)(kFftPoints64 * sizeof(double2));
    cudaError_t e = cudaFuncSetAttribute(fwd_rows64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cols64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(inv_rows64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

ws_status enqueue_grid64(ws_plan_s *p, const double *uvw, const double2 *vis, int64_t M, double2 *dirty,
                         cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(p->d_drop, 0, kCounters * sizeof(unsigned long long), s);
    const int64_t n_img = (int64_t)p->L.N * p->L.N;
    const size_t plane = (size_t)p->L.Np * p->L.Np;
    VisRec64 *rec = reinterpret_cast<VisRec64 *>(p->d_rec64);
    if (e == cudaSuccess && M > 0) {
        prep64_kernel<<<blocks64(M, 128), 128, 0, s>>>(p->L, uvw, M, rec, p->d_drop);
        e = cudaGetLastError();
    }
    for (int p0 = 0; p0 < p->L.Nw && e == cudaSuccess; p0 += p->planes64) {
        const int planes = std::min(p->planes64, p->L.Nw - p0);
        const Fft64Launch f(p->L, planes);
        e = cudaMemsetAsync(p->d_plane64, 0, planes * plane * sizeof(double2), s);
        if (e != cudaSuccess) break;
        if (M > 0)
            spread64_kernel<<<vis_blocks64(p, M), kThreads64, 0, s>>>(p->L, p->d_cheb64, p->fit.degree, rec, vis, M, p0,
                                                                       planes, p->d_plane64);
        cols64_kernel<<<f.cols, kFftThreads64, f.smem, s>>>(p->L, p->fft64_log, f.lines, p->d_tw64, 1, p->d_plane64);
        inv_rows64_kernel<<<f.rows, kFftThreads64, f.smem, s>>>(p->L, p->fft64_log, f.lines, p->d_tw64, p->d_z64, p0,
                                                               p->d_plane64);
        sum_planes64_kernel<<<blocks64(n_img, 128), 128, 0, s>>>(p->L, p->d_corr64, p->d_plane64, planes, p0 == 0,
                                                                p0 + planes == p->L.Nw, p->d_acc64, dirty);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? WS_OK : cuda_fail(e, "ws_grid (FP64 plan)");
}

ws_status enqueue_degrid64(ws_plan_s *p, const double2 *image, const double *uvw, int64_t M, double2 *vis,
                           cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(p->d_drop, 0, kCounters * sizeof(unsigned long long), s);
    if (M == 0) return e == cudaSuccess ? WS_OK : cuda_fail(e, "ws_degrid (FP64 plan)");
    VisRec64 *rec = reinterpret_cast<VisRec64 *>(p->d_rec64);
    if (e == cudaSuccess) e = cudaMemsetAsync(vis, 0, (size_t)M * sizeof(double2), s);
    if (e == cudaSuccess) {
        prep64_kernel<<<blocks64(M, 128), 128, 0, s>>>(p->L, uvw, M, rec, p->d_drop);
        e = cudaGetLastError();
    }
    for (int p0 = 0; p0 < p->L.Nw && e == cudaSuccess; p0 += p->planes64) {
        const int planes = std::min(p->planes64, p->L.Nw - p0);
        const Fft64Launch f(p->L, planes);
        fwd_rows64_kernel<<<f.rows, kFftThreads64, f.smem, s>>>(p->L, p->fft64_log, f.lines, p->d_tw64, p->d_corr64,
                                                               image, p->d_z64, p0, p->d_plane64);
        cols64_kernel<<<f.cols, kFftThreads64, f.smem, s>>>(p->L, p->fft64_log, f.lines, p->d_tw64, 0, p->d_plane64);
        gather64_kernel<<<vis_blocks64(p, M), kThreads64, 0, s>>>(p->L, p->d_cheb64, p->fit.degree, rec, M, p0, planes,
                                                                   p->d_plane64, vis);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        finish_degrid64_kernel<<<blocks64(M, 128), 128, 0, s>>>(rec, M, vis);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? WS_OK : cuda_fail(e, "ws_degrid (FP64 plan)");
}

}  // namespace ws
