// FFT engine for the w-plane transforms (Algorithm 5 step 3b, Algorithm 6
// step 3c).
//
// A CTA transforms one or two length-n sequences cooperatively with mixed-
// radix decimation in time, in place in shared memory.  The first stage reads
// its inputs straight from the caller (global memory, with zero padding and
// screens applied on the fly), transforms them in registers and scatters them
// to digit-reversed positions; every later stage reads, twiddles, transforms
// and writes back the same R positions, so a thread holds one butterfly at a
// time and a stage needs a single barrier; the last stage hands its outputs
// straight back (global stores, crops, accumulations).  Twiddles come from a
// table of exp(-2 pi i m / n) computed in double precision on the host.
//
// The forward and the inverse transforms of a size have plans of their own
// (fft_make_plan in plan.cpp).
//
// Shared-memory addressing inserts one pad slot after every `chunk` elements,
// which removes most bank conflicts of the digit-reversed scatter; two
// transforms of a CTA sit 8 (mod 16) slots apart so interleaved lanes use
// different banks.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fft_plan.hpp"
#include "packed.cuh"

namespace ws {

namespace fftdev {

template <int R>
struct Radix {
    static constexpr int value = R;
};

// exp(-+ 2 pi i m / n) from the forward table
__device__ __forceinline__ float2 twiddle(const float2 *__restrict__ tw, int m, bool inv) {
    float2 w = __ldg(tw + m);
    return inv ? make_float2(w.x, -w.y) : w;
}

// Powers of a butterfly's twiddle w: those its table holds (the others are not set).
struct Bases {
    float2 w1, w2, w4, w8;
};

// The bases of butterfly offset k of a runtime plan's stage of radix R, from row k of the
// stage's own table (fft_tables, base_row).
// Read from the N'-entry table, a warp's w^4k fell into as many sectors as
// lanes, and a stage's table is small enough for the L1 that the buffers leave.
template <int R, bool INV>
__device__ __forceinline__ Bases twiddle_bases(const float2 *__restrict__ bases, int k) {
    constexpr int ROW = base_row(R, INV);
    Bases b{};
    if constexpr (ROW == 1) {
        b.w1 = twiddle(bases, k, INV);
        return b;
    } else {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(bases + ROW * k));
        b.w1 = make_float2(w.x, INV ? -w.y : w.y);
        (INV ? b.w2 : b.w4) = make_float2(w.z, INV ? -w.w : w.w);
        if constexpr (ROW == 4 && R > 8) {
            const float4 h = __ldg(reinterpret_cast<const float4 *>(bases + ROW * k) + 1);
            b.w4 = make_float2(h.x, -h.y);
            b.w8 = make_float2(h.z, -h.w);
        } else if constexpr (ROW == 4) {
            b.w4 = twiddle(bases, ROW * k + 2, INV);
        }
        return b;
    }
}

__device__ __forceinline__ void dft4(float2 &a0, float2 &a1, float2 &a2, float2 &a3, bool inv) {
    const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), d = csub(a1, a3);
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    a1 = add_rot(t1, d, inv);
    a3 = sub_rot(t1, d, inv);
}

// the same with a2 to be taken times -i (forward) or +i (inverse) first
__device__ __forceinline__ void dft4_rot2(float2 &a0, float2 &a1, float2 &a2, float2 &a3, bool inv) {
    const float2 t0 = add_rot(a0, a2, inv), t1 = sub_rot(a0, a2, inv), t2 = cadd(a1, a3), d = csub(a1, a3);
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    a1 = add_rot(t1, d, inv);
    a3 = sub_rot(t1, d, inv);
}

// cos and sin of 2 pi m / 16 for m = 1, 2, 3 (exact decimal expansions)
constexpr float kC1 = 0.92387953251128674f;   // cos(pi/8)
constexpr float kS1 = 0.38268343236508978f;   // sin(pi/8)
constexpr float kR2 = 0.70710678118654752f;   // sqrt(1/2)

// a times exp(-+ 2 pi i m / 16), m = 1, 2, 3, 6 or 9 (products q*k1 of the 4x4 split; 4 is a quarter turn)
__device__ __forceinline__ float2 mul_w16(float2 a, int m, bool inv) {
    const float c = m == 1 ? kC1 : m == 2 ? kR2 : m == 3 ? kS1 : m == 6 ? -kR2 : -kC1;
    const float s = m == 1 ? kS1 : m == 2 ? kR2 : m == 3 ? kC1 : m == 6 ? kR2 : -kS1;
    return inv ? cmul_rot(a, make_float2(c, s), make_float2(-s, c))
               : cmul_rot(a, make_float2(c, -s), make_float2(s, c));
}

template <int R>
__device__ __forceinline__ void dft(float2 *v, bool inv);

template <>
__device__ __forceinline__ void dft<4>(float2 *v, bool inv) {
    dft4(v[0], v[1], v[2], v[3], inv);
}

template <>
__device__ __forceinline__ void dft<8>(float2 *v, bool inv) {
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4(e0, e1, e2, e3, inv);
    dft4(o0, o1, o2, o3, inv);
    o1 = mul_w16(o1, 2, inv);
    o3 = mul_w16(o3, 6, inv);
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1);
    v[5] = csub(e1, o1);
    v[2] = add_rot(e2, o2, inv);
    v[6] = sub_rot(e2, o2, inv);
    v[3] = cadd(e3, o3);
    v[7] = csub(e3, o3);
}

// Second level of the 4 x 4 split of radix 16: the twiddles w16^(q k1), then the
// 4-point DFTs over q, in natural output order.
__device__ __forceinline__ void dft16_second(float2 *v, bool inv) {
#pragma unroll
    for (int q = 1; q < 4; ++q)
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1)
            if (q * k1 != 4) v[q + 4 * k1] = mul_w16(v[q + 4 * k1], q * k1, inv);
    float2 o[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        float2 a0 = v[0 + 4 * k1], a1 = v[1 + 4 * k1], a2 = v[2 + 4 * k1], a3 = v[3 + 4 * k1];
        if (k1 == 2)
            dft4_rot2(a0, a1, a2, a3, inv);
        else
            dft4(a0, a1, a2, a3, inv);
        o[k1] = a0;
        o[k1 + 4] = a1;
        o[k1 + 8] = a2;
        o[k1 + 12] = a3;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = o[i];
}

template <>
__device__ __forceinline__ void dft<16>(float2 *v, bool inv) {
    // X[k1 + 4 k2] = sum_q w16^(q k1) w4^(q k2) sum_s v[q + 4 s] w4^(s k1)
#pragma unroll
    for (int q = 0; q < 4; ++q) dft4(v[q], v[q + 4], v[q + 8], v[q + 12], inv);
    dft16_second(v, inv);
}

// Radix 16 whose middle half of inputs, v[4] .. v[11], is zero (the centred
// half of a sequence of N' = 2N points zero-padded to N'): the first level's
// four 4-point DFTs see (a, 0, 0, d) and reduce to two adds and a quarter
// turn each; v[4..11] need not be set.
__device__ __forceinline__ void dft16_zero_middle(float2 *v, bool inv) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 a = v[q], d = v[q + 12];
        v[q] = cadd(a, d);
        v[q + 8] = csub(a, d);
        v[q + 4] = sub_rot(a, d, inv);
        v[q + 12] = add_rot(a, d, inv);
    }
    dft16_second(v, inv);
}

// cos and sin of 2 pi m / R for the odd radices R = 3, 5, 7 and 0 <= m < R
// (decimal expansions of the closed forms; sin is odd in m about R / 2).
__host__ __device__ constexpr double odd_cos(int R, int m) {
    const int k = m <= R / 2 ? m : R - m;
    return k == 0 ? 1.0
         : R == 3 ? -0.5
         : R == 5 ? (k == 1 ? 0.30901699437494742 : -0.80901699437494742)
         : (k == 1 ? 0.62348980185873353 : k == 2 ? -0.22252093395631440 : -0.90096886790241913);
}
__host__ __device__ constexpr double odd_sin(int R, int m) {
    const int k = m <= R / 2 ? m : R - m;
    const double s = k == 0 ? 0.0
                   : R == 3 ? 0.86602540378443865
                   : R == 5 ? (k == 1 ? 0.95105651629515357 : 0.58778525229247313)
                   : (k == 1 ? 0.78183148246802981 : k == 2 ? 0.97492791218182361 : 0.43388373911755812);
    return m <= R / 2 ? s : -s;
}

// Odd radix R = 2h + 1 in symmetric form.  With a_r = x_r + x_{R-r} and
// b_r = x_r - x_{R-r} (r = 1..h): X_0 = x_0 + sum a_r and, for k = 1..h,
// A_k = x_0 + sum_r cos(2 pi r k / R) a_r, B_k = sum_r sin(2 pi r k / R) b_r,
// X_k = A_k - i B_k and X_{R-k} = A_k + i B_k (the signs swap for the inverse).
template <int R>
__device__ __forceinline__ void dft_odd(float2 *v, bool inv) {
    constexpr int h = R / 2;
    float2 a[h + 1], b[h + 1];
#pragma unroll
    for (int r = 1; r <= h; ++r) {
        a[r] = cadd(v[r], v[R - r]);
        b[r] = csub(v[r], v[R - r]);
    }
    const float2 x0 = v[0];
    float2 s0 = x0;
#pragma unroll
    for (int r = 1; r <= h; ++r) s0 = cadd(s0, a[r]);
    v[0] = s0;
#pragma unroll
    for (int k = 1; k <= h; ++k) {
        float2 A = x0, B = make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 1; r <= h; ++r) {
            const float c = (float)odd_cos(R, (r * k) % R), sn = (float)odd_sin(R, (r * k) % R);
            A = fma2(a[r], dup2(c), A);
            B = r == 1 ? mul2(b[r], dup2(sn)) : fma2(b[r], dup2(sn), B);
        }
        v[k] = add_rot(A, B, inv);          // A - i B forward, A + i B inverse
        v[R - k] = sub_rot(A, B, inv);
    }
}
template <>
__device__ __forceinline__ void dft<3>(float2 *v, bool inv) {
    dft_odd<3>(v, inv);
}
template <>
__device__ __forceinline__ void dft<5>(float2 *v, bool inv) {
    dft_odd<5>(v, inv);
}
template <>
__device__ __forceinline__ void dft<7>(float2 *v, bool inv) {
    dft_odd<7>(v, inv);
}
template <>
__device__ __forceinline__ void dft<2>(float2 *v, bool) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
}

// R = A B with coprime A and B, by the prime factor form (Good, Thomas): with
// n = (B a + A b) mod R the kernel w_R^(n k) is w_A^(a k) w_B^(b k), so the DFT
// is an A x B two-dimensional one without twiddles; output k sits at (k mod A, k mod B).
template <int A, int B>
__device__ __forceinline__ void dft_pfa(float2 *v, bool inv) {
    float2 y[A][B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        float2 c[A];
#pragma unroll
        for (int a = 0; a < A; ++a) c[a] = v[(B * a + A * b) % (A * B)];
        dft<A>(c, inv);
#pragma unroll
        for (int a = 0; a < A; ++a) y[a][b] = c[a];
    }
#pragma unroll
    for (int a = 0; a < A; ++a) dft<B>(y[a], inv);
#pragma unroll
    for (int k = 0; k < A * B; ++k) v[k] = y[k % A][k % B];
}
template <>
__device__ __forceinline__ void dft<6>(float2 *v, bool inv) {
    dft_pfa<2, 3>(v, inv);
}
// Forward, radix 10 keeps the 5 x 2 form with the twiddles w10^k that it always had: the prime
// factor form, which the inverse takes, moved the model visibilities' error by up to 2 %
// (N' = 2560: 2.06e-7 -> 2.10e-7).
template <>
__device__ __forceinline__ void dft<10>(float2 *v, bool inv) {
    if (inv) {
        dft_pfa<2, 5>(v, true);
        return;
    }
    float2 e[5] = {v[0], v[2], v[4], v[6], v[8]}, o[5] = {v[1], v[3], v[5], v[7], v[9]};
    dft_odd<5>(e, false);
    dft_odd<5>(o, false);
    // cos and sin of 2 pi k / 10 from those of fifths of a turn
    constexpr float c[5] = {1.f, (float)-odd_cos(5, 2), (float)odd_cos(5, 1), (float)-odd_cos(5, 1), (float)odd_cos(5, 2)};
    constexpr float sn[5] = {0.f, (float)odd_sin(5, 2), (float)odd_sin(5, 1), (float)odd_sin(5, 1), (float)odd_sin(5, 2)};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const float2 t = k == 0 ? o[0] : cmul_rot(o[k], make_float2(c[k], -sn[k]), make_float2(sn[k], c[k]));
        v[k] = cadd(e[k], t);
        v[k + 5] = csub(e[k], t);
    }
}
template <>
__device__ __forceinline__ void dft<12>(float2 *v, bool inv) {
    dft_pfa<4, 3>(v, inv);
}
template <>
__device__ __forceinline__ void dft<14>(float2 *v, bool inv) {
    dft_pfa<2, 7>(v, inv);
}
template <>
__device__ __forceinline__ void dft<20>(float2 *v, bool inv) {
    dft_pfa<4, 5>(v, inv);
}
template <>
__device__ __forceinline__ void dft<21>(float2 *v, bool inv) {
    dft_pfa<3, 7>(v, inv);
}
template <>
__device__ __forceinline__ void dft<28>(float2 *v, bool inv) {
    dft_pfa<4, 7>(v, inv);
}
template <>
__device__ __forceinline__ void dft<24>(float2 *v, bool inv) {
    dft_pfa<8, 3>(v, inv);
}

// A twiddle and the pair its products need.
struct Tw {
    float2 w, rot;
    __device__ __forceinline__ explicit Tw(float2 v) : w(v), rot(turn2(v)) {}
    __device__ __forceinline__ float2 times(float2 a) const { return cmul_rot(a, w, rot); }
};

// v[m] *= w^m for m = 1..R-1, w = exp(-+ 2 pi i e / n), given the powers that
// base_row<R, INV> names.  The table holds w^m to half an ulp, but a warp's loads of
// w^m for m > 1 scatter over many sectors; so only those powers are read and the
// others are products of them (forward, at most five roundings: RMS error about 7e-8
// against 2e-8 for the table).
template <int R, bool INV>
__device__ __forceinline__ void twiddle_powers(float2 *v, const Bases &b) {
    static_assert(R >= 3 && R <= 21, "powers up to w^20");
    constexpr bool W4 = base_row(R, INV) == (INV ? 4 : 2), W8 = base_row(R, INV) == 4;
    const Tw t1(b.w1);
    v[1] = t1.times(v[1]);
    const Tw t2(INV ? b.w2 : t1.times(b.w1));
    v[2] = t2.times(v[2]);
    if constexpr (R >= 4) {
        const Tw t3(t1.times(t2.w));
        v[3] = t3.times(v[3]);
        if constexpr (R > 4) {
            const Tw t4(W4 ? b.w4 : t2.times(t2.w));
            float2 base = t4.w, w8 = t4.w;
#pragma unroll
            for (int a = 1; 4 * a < R; ++a) {
                if (a == 2) base = w8 = W8 ? b.w8 : t4.times(t4.w);
                if (a == 3 || a == 5) base = t4.times(base);
                if (a == 4) base = Tw(w8).times(w8);
                v[4 * a] = Tw(base).times(v[4 * a]);
                if (4 * a + 1 < R) v[4 * a + 1] = Tw(t1.times(base)).times(v[4 * a + 1]);
                if (4 * a + 2 < R)
                    v[4 * a + 2] = Tw(R == 7 && !W4 ? t3.times(t3.w) : t2.times(base)).times(v[4 * a + 2]);
                if (4 * a + 3 < R) v[4 * a + 3] = Tw(t3.times(base)).times(v[4 * a + 3]);
            }
        }
    }
}
// The same with w and, from R = 8 on, w^4 given, as the compile-time plans keep them in either direction.
template <int R>
__device__ __forceinline__ void twiddle_powers(float2 *v, float2 w1, float2 w4) {
    Bases b{};
    b.w1 = w1;
    b.w4 = w4;
    twiddle_powers<R, false>(v, b);
}

// x / d for 0 <= x < 2^16, 1 <= d < 2^13, with mul = div_mul(d) (fft_plan.hpp)
__device__ __forceinline__ int div_small(int x, unsigned mul) {
    return mul ? (int)__umulhi((unsigned)x, mul) : x;
}

// In-place decimation-in-time stage of radix R: for every block b of R*L
// positions and offset k < L, the R elements at b*R*L + k + m*L (m < R) are
// multiplied by w_{RL}^{k m}, transformed by an R-point DFT and written back
// to the same positions.  Butterflies own disjoint positions, so a thread
// can do them one after another and a stage needs no barrier between its
// reads and writes.  Work item q -> transform t = q % COUNT, butterfly q / COUNT.
//
// A butterfly's slots are one base plus multiples of P.step[s] (FftPlan), so the
// slot arithmetic costs once per butterfly.
//
// The barrier that completes the previous stage comes after the first round's
// twiddles have been asked for, and each round asks for the next one's: the table
// mostly comes from L2 (the buffers leave little L1), and a stage that waited for
// it after the barrier spent a third of its time there.
template <int R, int COUNT, bool LAST, bool INV, class Store>
__device__ __forceinline__ void dit_stage(float2 *buf, const FftPlan &P, int s, const float2 *__restrict__ tw, int tid,
                                          int nthr, Store &store) {
    const int L = P.L[s], total = COUNT * P.nb[s], step = P.step[s];
    tw += P.bases[s];
    Bases w{};
    int base = 0, k = 0;
    auto fetch = [&](int q) {                // butterfly q's first position and twiddles (past the end: the last one's)
        const int bq = min(q, total - 1) / COUNT;
        const int blk = LAST ? 0 : div_small(bq, P.L_mul[s]);
        k = bq - blk * L;
        base = blk * R * L + k;
        w = twiddle_bases<R, INV>(tw, k);
    };
    fetch(tid);
    __syncthreads();
    for (int q = tid; q < total; q += nthr) {
        const int t = q % COUNT, b = base, kq = k;
        const Bases wq = w;
        float2 *x = buf + t * P.stride + b + div_small(b, P.chunk_mul);
        float2 v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = x[m * step];
        fetch(q + nthr);
        if (kq > 0) twiddle_powers<R, INV>(v, wq);
        dft<R>(v, INV);
        if constexpr (LAST) {
            store(std::false_type{}, t, b, L, v);
        } else {
#pragma unroll
            for (int m = 0; m < R; ++m) x[m * step] = v[m];
        }
    }
}

// Stages s (radix A) and s + 1 (radix B) in one pass: a thread holds the A B
// elements k + m1 L + m2 A L of a block, does the B butterflies of the first stage
// and then the A butterflies of the second, whose twiddles are those of k + m1 L.
// For one transform (the rows; for the columns' pairs it was slower: N' = 2016, rows
// 746 -> 650 us, columns 856 -> 896, on 68 planes).
// The arithmetic is that of the two stages; one trip through shared memory and one
// barrier less.
template <int A, int B, bool LAST, class Store>
__device__ __forceinline__ void dit_pair(float2 *buf, const FftPlan &P, int s, const float2 *__restrict__ tw, int tid,
                                         int nthr, Store &store) {
    constexpr bool inv = false;
    static_assert(B < 8, "the second radix takes its twiddles from w alone");
    const int L = P.L[s], total = P.nb[s] / B, step_a = P.step[s], step_b = P.step[s + 1];
    Bases w_a{};
    int base = 0, k = 0;
    auto fetch = [&](int q) {                // as in dit_stage, for the first of the two stages
        const int bq = min(q, total - 1);
        const int blk = LAST ? 0 : div_small(bq, P.L_mul[s]);
        k = bq - blk * L;
        base = blk * A * B * L + k;
        w_a = twiddle_bases<A, inv>(tw + P.bases[s], k);
    };
    fetch(tid);
    __syncthreads();
    for (int q = tid; q < total; q += nthr) {
        const int b = base, kq = k;
        const Bases wq = w_a;
        float2 *x = buf + b + div_small(b, P.chunk_mul);
        float2 v[A * B], w[A];
#pragma unroll
        for (int m1 = 0; m1 < A; ++m1) w[m1] = twiddle(tw + P.bases[s + 1], kq + m1 * L, inv);
#pragma unroll
        for (int m2 = 0; m2 < B; ++m2)
#pragma unroll
            for (int m1 = 0; m1 < A; ++m1) v[m1 + A * m2] = x[m1 * step_a + m2 * step_b];
        fetch(q + nthr);
#pragma unroll
        for (int m2 = 0; m2 < B; ++m2) {
            if (kq > 0) twiddle_powers<A, inv>(v + A * m2, wq);
            dft<A>(v + A * m2, inv);
        }
#pragma unroll
        for (int m1 = 0; m1 < A; ++m1) {
            float2 c[B];
#pragma unroll
            for (int m2 = 0; m2 < B; ++m2) c[m2] = v[m1 + A * m2];
            if (m1 > 0 || kq > 0) twiddle_powers<B>(c, w[m1], w[m1]);
            dft<B>(c, inv);
#pragma unroll
            for (int m2 = 0; m2 < B; ++m2) v[m1 + A * m2] = c[m2];
        }
        if constexpr (LAST) {
            store(std::false_type{}, 0, b, L, v);
        } else {
#pragma unroll
            for (int m2 = 0; m2 < B; ++m2)
#pragma unroll
                for (int m1 = 0; m1 < A; ++m1) x[m1 * step_a + m2 * step_b] = v[m1 + A * m2];
        }
    }
}

// The last stage of one transform, its inputs all read before between() runs
// (the buffer is free from then on): up to ROUNDS butterflies a thread in
// registers, R ROUNDS <= 32.
template <int R, class Between, class Store>
__device__ __forceinline__ void dit_last_held(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw, int tid,
                                              int nthr, Between &between, Store &store) {
    constexpr bool inv = true;
    constexpr int ROUNDS = 32 / R;
    const int s = P.nstages - 1, L = P.L[s], nb = P.nb[s], step = P.step[s];
    float2 v[ROUNDS][R];
    Bases w[ROUNDS];
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
        w[i] = twiddle_bases<R, inv>(tw + P.bases[s], min(tid + i * nthr, nb - 1));
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
        const int k = min(tid + i * nthr, nb - 1);
        const float2 *x = buf + k + div_small(k, P.chunk_mul);
#pragma unroll
        for (int m = 0; m < R; ++m) v[i][m] = x[m * step];
    }
    __syncthreads();
    between();
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
        const int k = tid + i * nthr;
        if (k >= nb) break;
        if (k > 0) twiddle_powers<R, inv>(v[i], w[i]);
        dft<R>(v[i], inv);
        store(std::false_type{}, 0, k, L, v[i]);
    }
}

// The slot where butterfly j of the first stage puts its R outputs: that of
// position g*R, g = the digits of j in reverse order (from the plan's table: the
// digits took a dozen instructions per stage, five per element of a radix-8 stage).
__device__ __forceinline__ int first_slot(const FftPlan &P, const float2 *__restrict__ tw, int j) {
    return __ldg(reinterpret_cast<const int *>(tw) + P.slots + j);
}

// First stage: butterfly j of each transform reads inputs m*(n/R) + j, m < R,
// straight from load(t, e), and writes them to the digit-reversed positions
// g*R + m that the later in-place stages expect.
template <int R, int COUNT, class Load>
__device__ __forceinline__ void dit_first(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw, bool inv,
                                          int tid, int nthr, Load &load) {
    const int nb = P.nb[0], total = COUNT * nb;
    for (int q = tid; q < total; q += nthr) {
        const int t = q % COUNT, j = q / COUNT;
        const int slot = first_slot(P, tw, j);
        float2 v[R];
        load(std::false_type{}, t, j, nb, v);
        dft<R>(v, inv);
        float2 *x = buf + t * P.stride + slot;
#pragma unroll
        for (int m = 0; m < R; ++m) x[m] = v[m];
    }
}

// First stage of one transform whose input sits in the buffer in natural order
// at 0..n-1 (n / R <= nthr: one butterfly per thread); input m of a thread is
// zero where bit m of live is clear, whatever the buffer holds.
template <int R>
__device__ __forceinline__ void dit_first_inplace(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw,
                                                  bool inv, int tid, uint32_t live) {
    // threads past nb read the last butterfly's inputs and drop them: a value that
    // exists only under a condition, kept across the barrier, made the compiler spill
    const int nb = P.nb[0], at = min(tid, nb - 1), slot = first_slot(P, tw, at);
    float2 v[R];
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const float2 x = buf[m * nb + at];
        v[m] = (live >> m) & 1u ? x : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (tid < nb) {
        dft<R>(v, inv);
        float2 *x = buf + slot;
#pragma unroll
        for (int m = 0; m < R; ++m) x[m] = v[m];
    }
}

// Calls f(Radix<r>) for the first or a later radix of a forward plan, and for the
// first, a middle or the last radix of an inverse plan (the sets that
// fft_make_plan chooses from).
template <class F>
__device__ __forceinline__ void with_forward_first(int r, F f) {
    if (r == 16)
        f(Radix<16>{});
    else
        f(Radix<8>{});
}
template <class F>
__device__ __forceinline__ void with_forward_later(int r, F f) {
    switch (r) {
        case 16: f(Radix<16>{}); break;
        case 10: f(Radix<10>{}); break;
        case 8: f(Radix<8>{}); break;
        case 7: f(Radix<7>{}); break;
        case 5: f(Radix<5>{}); break;
        case 4: f(Radix<4>{}); break;
        default: f(Radix<3>{}); break;
    }
}
// The pairs of consecutive forward radices that run as one pass (fft_make_plan): f(Radix<A>, Radix<B>).
template <class F>
__device__ __forceinline__ void with_forward_pair(int a, int b, F f) {
    switch (16 * a + b) {
        case 16 * 4 + 7: f(Radix<4>{}, Radix<7>{}); break;
        case 16 * 4 + 3: f(Radix<4>{}, Radix<3>{}); break;
        case 16 * 7 + 3: f(Radix<7>{}, Radix<3>{}); break;
        case 16 * 5 + 5: f(Radix<5>{}, Radix<5>{}); break;
        case 16 * 5 + 3: f(Radix<5>{}, Radix<3>{}); break;
        case 16 * 8 + 3: f(Radix<8>{}, Radix<3>{}); break;
        default: f(Radix<3>{}, Radix<3>{}); break;
    }
}
template <class F>
__device__ __forceinline__ void with_first_radix(int r, F f) {
    switch (r) {
        case 28: f(Radix<28>{}); break;
        case 24: f(Radix<24>{}); break;
        case 20: f(Radix<20>{}); break;
        case 16: f(Radix<16>{}); break;
        case 14: f(Radix<14>{}); break;
        case 12: f(Radix<12>{}); break;
        case 10: f(Radix<10>{}); break;
        default: f(Radix<8>{}); break;
    }
}
template <class F>
__device__ __forceinline__ void with_middle_radix(int r, F f) {
    switch (r) {
        case 21: f(Radix<21>{}); break;
        case 20: f(Radix<20>{}); break;
        case 16: f(Radix<16>{}); break;
        case 14: f(Radix<14>{}); break;
        case 12: f(Radix<12>{}); break;
        case 10: f(Radix<10>{}); break;
        case 8: f(Radix<8>{}); break;
        default: f(Radix<6>{}); break;
    }
}
template <class F>
__device__ __forceinline__ void with_last_radix(int r, F f) {
    switch (r) {
        case 16: f(Radix<16>{}); break;
        case 14: f(Radix<14>{}); break;
        case 12: f(Radix<12>{}); break;
        case 10: f(Radix<10>{}); break;
        case 8: f(Radix<8>{}); break;
        case 7: f(Radix<7>{}); break;
        case 6: f(Radix<6>{}); break;
        default: f(Radix<4>{}); break;
    }
}

}  // namespace fftdev

// Transform COUNT sequences of length P.n, using the shared buffers buf + t * P.stride between stages.
// All threads of the CTA must call it; shared buffers may be reused after the
// caller's next barrier.
// The stages between the first and the last pass; returns the last pass's (first) stage.
template <int COUNT, bool INV>
__device__ __forceinline__ int fft_middle_stages(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw, int tid,
                                                 int nthr) {
    auto none = [](auto, int, int, int, auto &) {};
    int s = 1;
    auto fused = [&](int i) { return COUNT == 1 && !INV ? P.fuse[i] : 0; };     // rows only (FftPlan)
    while (s + fused(s) < P.nstages - 1) {
        auto stage = [&](auto r) {
            fftdev::dit_stage<decltype(r)::value, COUNT, false, INV>(buf, P, s, tw, tid, nthr, none);
        };
        if constexpr (INV) {
            fftdev::with_middle_radix(P.radix[s], stage);
        } else if (fused(s)) {
            if constexpr (COUNT == 1)
                fftdev::with_forward_pair(P.radix[s], P.radix[s + 1], [&](auto ra, auto rb) {
                    fftdev::dit_pair<decltype(ra)::value, decltype(rb)::value, false>(buf, P, s, tw, tid, nthr, none);
                });
        } else {
            fftdev::with_forward_later(P.radix[s], stage);
        }
        s += 1 + fused(s);
    }
    return s;
}

template <int COUNT, bool INV, class Store>
__device__ __forceinline__ void fft_last_stage(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw, int last,
                                               int tid, int nthr, Store &store) {
    auto stage = [&](auto r) {
        fftdev::dit_stage<decltype(r)::value, COUNT, true, INV>(buf, P, last, tw, tid, nthr, store);
    };
    if constexpr (INV) {
        fftdev::with_last_radix(P.radix[last], stage);
    } else {
        if constexpr (COUNT == 1)
            if (P.fuse[last]) {
                fftdev::with_forward_pair(P.radix[last], P.radix[last + 1], [&](auto ra, auto rb) {
                    fftdev::dit_pair<decltype(ra)::value, decltype(rb)::value, true>(buf, P, last, tw, tid, nthr, store);
                });
                return;
            }
        fftdev::with_forward_later(P.radix[last], stage);
    }
}

//
// load(t, e0, step, v) fills a first-stage butterfly's inputs v[m], element e0 +
// m step of transform t (t < COUNT), and store(t, e0, step, v) takes a last-stage
// butterfly's outputs; both get a whole butterfly, so that what they read from
// shared memory is under way before what they write (element by element, each
// read waited for the write before it).  Under PRUNE_IN / PRUNE_OUT only the
// first and last quarter of v counts (first argument: whether that is so).
template <int COUNT, bool INV, class Load, class Store>
__device__ __forceinline__ void fft_many(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw, int tid,
                                         int nthr, Load load, Store store) {
    auto first = [&](auto r) {
        fftdev::dit_first<decltype(r)::value, COUNT>(buf, P, tw, INV, tid, nthr, load);
    };
    if constexpr (INV)
        fftdev::with_first_radix(P.radix[0], first);
    else
        fftdev::with_forward_first(P.radix[0], first);
    const int last = fft_middle_stages<COUNT, INV>(buf, P, tw, tid, nthr);
    fft_last_stage<COUNT, INV>(buf, P, tw, last, tid, nthr, store);
}

// One inverse transform whose input sits in buf in natural order (see
// dit_first_inplace).  HELD: between() runs once the buffer's last contents are
// read (the plan's last stage has at most 32 / radix rounds).
template <bool HELD, class Between, class Store>
__device__ __forceinline__ void fft_inplace(float2 *buf, const FftPlan &P, const float2 *__restrict__ tw, int tid,
                                            int nthr, Between between, Store store, uint32_t live) {
    fftdev::with_first_radix(P.radix[0], [&](auto r) {
        fftdev::dit_first_inplace<decltype(r)::value>(buf, P, tw, true, tid, live);
    });
    const int last = fft_middle_stages<1, true>(buf, P, tw, tid, nthr);
    if constexpr (HELD)
        fftdev::with_last_radix(P.radix[last], [&](auto r) {
            fftdev::dit_last_held<decltype(r)::value>(buf, P, tw, tid, nthr, between, store);
        });
    else
        fft_last_stage<1, true>(buf, P, tw, last, tid, nthr, store);
}

// -- compile-time plans for the power-of-two sizes -----------------------------
//
// For N' = 512, 1024, 2048 and 4096 the radix sequence, the digit weights of
// the first stage, the padding and every stride are constants, so each padded
// shared-memory address is one base plus an immediate offset and each
// twiddle index is one multiply.  The layout and the arithmetic are those of
// the runtime engine above (same stride and padding), only specialised.

namespace fftst {

__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v / 2); }

template <int N> struct Radices;
template <> struct Radices<4096> { static constexpr int n = 3, r0 = 16, r1 = 16, r2 = 16; };
template <> struct Radices<2048> { static constexpr int n = 3, r0 = 16, r1 = 16, r2 = 8; };
template <> struct Radices<1024> { static constexpr int n = 3, r0 = 16, r1 = 8, r2 = 8; };
template <> struct Radices<512> { static constexpr int n = 3, r0 = 16, r1 = 8, r2 = 4; };

template <int N> struct Layout {
    static constexpr int shift = ilog2(N / Radices<N>::r0) < 4 ? 4 : ilog2(N / Radices<N>::r0);
    static constexpr int len = (N - 1) + ((N - 1) >> shift) + 1;
    static constexpr int stride = len + ((8 - len % 16) + 16) % 16;
    __host__ __device__ static constexpr int pad(int e) { return e + (e >> shift); }
};

// Crop pruning (N' = 2N, the centred half of a sequence is the crop): PRUNE_IN
// when the inputs outside it are zero, PRUNE_OUT when the outputs outside it
// are not wanted.  In the first stage, input m (N/R0) + j lies outside it for
// R0/4 <= m < 3 R0/4; in the last stage, output k + m (N/R) likewise.
constexpr int PRUNE_IN = 1, PRUNE_OUT = 2;

// First stage (radix R0) of COUNT transforms by T threads: inputs m*(N/R0) + j, outputs to digit-reversed g*R0 + m.
template <int N, int COUNT, int T, int PRUNE, class Load>
__device__ __forceinline__ void first(float2 *buf, bool inv, int tid, Load &load) {
    using Rd = Radices<N>;
    using Ly = Layout<N>;
    constexpr int R = Rd::r0, nb = N / R, total = COUNT * nb;
    constexpr bool pin = (PRUNE & PRUNE_IN) != 0;
    static_assert(!pin || R == 16, "input pruning is written for a radix-16 first stage");
    // j = d1 * r2 + d2 (x-order); g = d1 + d2 * r1 (position order)
    for (int q = tid; q < total; q += T) {
        const int t = q % COUNT, j = q / COUNT;
        float2 v[R];
        load(std::bool_constant<pin>{}, t, j, nb, v);
        if constexpr (pin)
            fftdev::dft16_zero_middle(v, inv);
        else
            fftdev::dft<R>(v, inv);
        const int d1 = j >> ilog2(Rd::r2), d2 = j & (Rd::r2 - 1);
        const int g = d1 + d2 * Rd::r1;
        float2 *x = buf + t * Ly::stride + Ly::pad(g * R);     // R divides 2^shift: one base
#pragma unroll
        for (int m = 0; m < R; ++m) x[m] = v[m];
    }
}

// Twiddle bases w, w^4 of the butterflies a thread owns in a later stage of one
// transform by T threads (butterflies tid + i T): they do not change from
// transform to transform, so a kernel that loops over many transforms reads
// them once.  Where T is a multiple of L every round has the same ones.
template <int N, int R, int L, int T>
struct StageTw {
    static constexpr int rounds = (N / R + T - 1) / T, kept = T % L == 0 ? 1 : rounds;
    float2 w1[kept], w4[kept];
    __device__ __forceinline__ void load(const float2 *__restrict__ tw, bool inv, int tid) {
        constexpr int lgtw = ilog2(N / (R * L));
#pragma unroll
        for (int i = 0; i < kept; ++i) {
            const int k = (tid + i * T) & (L - 1);
            w1[i] = fftdev::twiddle(tw, k << lgtw, inv);
            w4[i] = R >= 8 ? fftdev::twiddle(tw, (4 * k) << lgtw, inv) : make_float2(1.f, 0.f);
        }
    }
};
struct NoTw {};

// Later stage of radix R over span L (constants) of COUNT transforms by T
// threads: in place, or to store() if LAST.  PRE holds the thread's twiddle
// bases (COUNT = 1), or is NoTw.
template <int N, int COUNT, int T, int R, int L, bool LAST, int PRUNE, class Pre, class Store>
__device__ __forceinline__ void later(float2 *buf, const float2 *__restrict__ tw, bool inv, int tid, const Pre &pre,
                                      Store &store) {
    constexpr bool pout = LAST && (PRUNE & PRUNE_OUT) != 0;
    static_assert(!pout || (R % 4 == 0 && R * L == N), "output pruning needs the last stage, R a multiple of 4");
    constexpr bool kept_tw = !std::is_same<Pre, NoTw>::value;
    static_assert(!kept_tw || COUNT == 1, "kept twiddle bases belong to one transform");
    using Ly = Layout<N>;
    constexpr int nb = N / R, total = COUNT * nb, rounds = (total + T - 1) / T;
    constexpr int lgL = ilog2(L), lgtw = ilog2(N / (R * L));
    // pad(base + m L) with base = blk R L + k, k < L, is pad_base + m * step when
    //  (a) L is a multiple of 2^shift (the pad of m L is exact), or
    //  (b) R L divides 2^shift ((blk R L + k + m L) >> shift = (blk R L) >> shift);
    // otherwise each element is padded on its own.
    constexpr bool wide = (L >> Ly::shift) > 0;
    constexpr bool inblock = (R * L) <= (1 << Ly::shift);
    constexpr bool affine = wide || inblock;
    constexpr int step = wide ? L + (L >> Ly::shift) : L;
    auto at = [&](int pbase, int base, int m) {
        return affine ? pbase + m * step : Ly::pad(base + m * L);
    };
    // the previous stage is complete after the barrier; twiddles that are not kept
    // are asked for before it, the next round's ahead of this one's arithmetic
    float2 w1, w4;
    auto fetch = [&](int i) {
        const int e = ((min(tid + i * T, total - 1) / COUNT) & (L - 1)) << lgtw;
        w1 = fftdev::twiddle(tw, e, inv);
        w4 = R >= 8 ? fftdev::twiddle(tw, 4 * e, inv) : make_float2(1.f, 0.f);
    };
    if constexpr (!kept_tw) fetch(0);
    __syncthreads();
#pragma unroll(kept_tw ? rounds : 1)
    for (int i = 0; i < rounds; ++i) {
        const int q = tid + i * T;
        if (total % T != 0 && q >= total) break;
        const int t = q % COUNT, bq = q / COUNT;
        const int blk = bq >> lgL, k = bq & (L - 1);
        const int base = blk * R * L + k;
        const int pbase = wide ? Ly::pad(base) : base + ((blk * R * L) >> Ly::shift);
        float2 *x = buf + t * Ly::stride;
        float2 v[R], v1, v4;
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = x[at(pbase, base, m)];
        if constexpr (kept_tw) {
            v1 = pre.w1[Pre::kept == 1 ? 0 : i];
            v4 = pre.w4[Pre::kept == 1 ? 0 : i];
        } else {
            v1 = w1;
            v4 = w4;
            if (i + 1 < rounds) fetch(i + 1);
        }
        if (k > 0) fftdev::twiddle_powers<R>(v, v1, v4);
        fftdev::dft<R>(v, inv);
        if constexpr (LAST) {
            store(std::bool_constant<pout>{}, t, base, L, v);
        } else {
#pragma unroll
            for (int m = 0; m < R; ++m) x[at(pbase, base, m)] = v[m];
        }
    }
}

// The last stage of one transform with all its inputs read before between() runs
// (the buffer is free from then on).
template <int N, int T, int R, int L, int PRUNE, class Pre, class Between, class Store>
__device__ __forceinline__ void last_held(float2 *buf, int tid, bool inv, const Pre &pre, Between &between,
                                          Store &store) {
    constexpr bool pout = (PRUNE & PRUNE_OUT) != 0;
    using Ly = Layout<N>;
    constexpr int rounds = N / R / T;
    static_assert(R * L == N && rounds * T * R == N && (L >> Ly::shift) > 0, "a last stage in whole rounds");
    constexpr int step = L + (L >> Ly::shift);
    float2 v[rounds][R];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < rounds; ++i)
#pragma unroll
        for (int m = 0; m < R; ++m) v[i][m] = buf[Ly::pad(tid + i * T) + m * step];
    __syncthreads();
    between();
#pragma unroll
    for (int i = 0; i < rounds; ++i) {
        const int k = tid + i * T;
        if (k > 0) fftdev::twiddle_powers<R>(v[i], pre.w1[Pre::kept == 1 ? 0 : i], pre.w4[Pre::kept == 1 ? 0 : i]);
        fftdev::dft<R>(v[i], inv);
        store(std::bool_constant<pout>{}, 0, k, L, v[i]);
    }
}

// First stage for inputs already in the buffer, in natural order at 0..N-1
// (one transform, N / R0 threads).  Each thread reads the R0 inputs m (N/R0) +
// tid (input m is zero where bit m of live is clear, whatever the buffer holds),
// the CTA synchronises, and the outputs go to their padded digit-reversed slots.
template <int N>
__device__ __forceinline__ void first_inplace(float2 *buf, bool inv, int tid, uint32_t live) {
    using Rd = Radices<N>;
    using Ly = Layout<N>;
    constexpr int R = Rd::r0, nb = N / R;
    float2 v[R];
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const float2 x = buf[m * nb + tid];
        v[m] = (live >> m) & 1u ? x : make_float2(0.f, 0.f);
    }
    __syncthreads();
    fftdev::dft<R>(v, inv);
    const int d1 = tid >> ilog2(Rd::r2), d2 = tid & (Rd::r2 - 1);
    float2 *x = buf + Ly::pad((d1 + d2 * Rd::r1) * R);
#pragma unroll
    for (int m = 0; m < R; ++m) x[m] = v[m];
}

// Twiddle bases of both later stages of one transform by T threads.
template <int N, int T>
struct RowTw {
    using Rd = Radices<N>;
    StageTw<N, Rd::r1, Rd::r0, T> s2;
    StageTw<N, Rd::r2, Rd::r0 * Rd::r1, T> s3;
    __device__ __forceinline__ RowTw(const float2 *__restrict__ tw, bool inv, int tid) {
        s2.load(tw, inv, tid);
        s3.load(tw, inv, tid);
    }
};

// -- two-stage transforms of 4096 = 64 x 64 points ------------------------------
//
// A thread transforms 64 points in registers (128 of them), so a sequence goes
// through shared memory once instead of twice and a CTA has one barrier:
//   X[k1 + 64 k2] = sum_j w64^(j k2) w4096^(j k1) sum_m x[j + 64 m] w64^(m k1)
// with thread j in the first stage and thread k1 in the second.  Radix 64 is 8 x 8.

// cos and sin of 2 pi m / 64 for m = 0..63 (decimal expansions over an eighth of the circle)
__host__ __device__ constexpr double cos64(int m) {
    constexpr double c[9] = {1.0, 0.99518472667219688624, 0.98078528040323044913, 0.95694033573220886494,
                             0.92387953251128675613, 0.88192126434835502971, 0.83146961230254523708,
                             0.77301045336273696081, 0.70710678118654752440};
    constexpr double s[9] = {0.0, 0.09801714032956060199, 0.19509032201612826785, 0.29028467725446236764,
                             0.38268343236508977173, 0.47139673682599764856, 0.55557023301960222474,
                             0.63439328416364549822, 0.70710678118654752440};
    const int r = m & 63, q = r >= 32 ? 64 - r : r;                  // cos is even about 0 and 32
    const int h = q > 16 ? 32 - q : q;                               // and odd about 16
    const double v = h <= 8 ? c[h] : s[16 - h];
    return q > 16 ? -v : v;
}
__host__ __device__ constexpr double sin64(int m) { return cos64(m + 48); }

// v[8 b + q] *= w64^(b q), forward or inverse, for the constants of one b
template <int B, int Q = 1>
__device__ __forceinline__ void mul_w64(float2 *v, bool inv) {
    if constexpr (Q < 8) {
        constexpr float c = (float)cos64(B * Q), s = (float)sin64(B * Q);
        v[8 * B + Q] = inv ? cmul_rot(v[8 * B + Q], make_float2(c, s), make_float2(-s, c))
                           : cmul_rot(v[8 * B + Q], make_float2(c, -s), make_float2(s, c));
        mul_w64<B, Q + 1>(v, inv);
    }
}
template <int B = 1>
__device__ __forceinline__ void mul_w64_all(float2 *v, bool inv) {
    if constexpr (B < 8) {
        mul_w64<B>(v, inv);
        mul_w64_all<B + 1>(v, inv);
    }
}

// 8-point DFT of (a0, a1, 0, 0, 0, 0, a6, a7) (v[2..5] need not be set)
__device__ __forceinline__ void dft8_zero_middle(float2 *v, bool inv) {
    // even inputs (v0, 0, 0, v6), odd inputs (v1, 0, 0, v7)
    const float2 e0 = cadd(v[0], v[6]), e2 = csub(v[0], v[6]);
    const float2 e1 = sub_rot(v[0], v[6], inv), e3 = add_rot(v[0], v[6], inv);
    const float2 o0 = cadd(v[1], v[7]), o2 = csub(v[1], v[7]);
    const float2 o1 = fftdev::mul_w16(sub_rot(v[1], v[7], inv), 2, inv);
    const float2 o3 = fftdev::mul_w16(add_rot(v[1], v[7], inv), 6, inv);
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1);
    v[5] = csub(e1, o1);
    v[2] = add_rot(e2, o2, inv);
    v[6] = sub_rot(e2, o2, inv);
    v[3] = cadd(e3, o3);
    v[7] = csub(e3, o3);
}

// In-register 64-point DFT: v[8 a + b], a, b < 8, becomes output q + 8 p in v[8 q + p].
// PIN: only a = 0, 1, 6, 7 are non-zero (the others need not be set).
template <bool PIN>
__device__ __forceinline__ void dft64_over_a(float2 *v, bool inv) {
    float2 o[64];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        float2 c[8];
#pragma unroll
        for (int a = 0; a < 8; ++a)
            if (!PIN || a < 2 || a > 5) c[a] = v[8 * a + b];
        if constexpr (PIN)
            dft8_zero_middle(c, inv);
        else
            fftdev::dft<8>(c, inv);
#pragma unroll
        for (int q = 0; q < 8; ++q) o[8 * b + q] = c[q];
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = o[i];           // v[8 b + q]
}
__device__ __forceinline__ void dft64_over_b(float2 *v, bool inv) {
    mul_w64_all(v, inv);
    float2 o[64];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        float2 c[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) c[b] = v[8 * b + q];
        fftdev::dft<8>(c, inv);
#pragma unroll
        for (int p = 0; p < 8; ++p) o[8 * q + p] = c[p];
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = o[i];
}

// v[8 r + i] *= w^r for r = 1..7, all i, given w, w^2 and w^4: the other powers are
// products of these.  (All powers from w alone multiplied its rounding error by up to
// seven: error against the exact DFT 3.3e-7 on the survey against 3.1e-7.)
__device__ __forceinline__ void mul_rows(float2 *v, const float2 (&w)[3]) {
    const fftdev::Tw t1(w[0]), t2(w[1]), t4(w[2]);
    auto row = [&](int r, const fftdev::Tw &t) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[8 * r + i] = t.times(v[8 * r + i]);
    };
    row(1, t1);
    row(2, t2);
    row(4, t4);
    row(5, fftdev::Tw(t1.times(t4.w)));
    row(6, fftdev::Tw(t2.times(t4.w)));
    const fftdev::Tw t3(t1.times(t2.w));
    row(3, t3);
    row(7, fftdev::Tw(t3.times(t4.w)));
}

constexpr int kPitch64 = 65;                             // row pitch of the exchange, in points
constexpr int kStride64 = 64 * kPitch64 + 8;             // points per sequence; 8 (mod 16)

}  // namespace fftst

// COUNT sequences of 4096 points by 64 COUNT threads (load and store as for
// fft_many, 64 points each; under PRUNE_IN / PRUNE_OUT the first and last quarter).
// bases: w^j, w^2j, .. w^32j for each j < 64 (fft_tables).
template <int COUNT, int PRUNE, class Load, class Store>
__device__ __forceinline__ void fft_4096_two_stage(float2 *buf, const float2 *__restrict__ bases, bool inv, int tid,
                                                   Load load, Store store) {
    using namespace fftst;
    const int t = tid % COUNT, j = tid / COUNT;
    float2 *x = buf + t * kStride64;
    float2 v[64];
    load(std::bool_constant<(PRUNE & PRUNE_IN) != 0>{}, t, j, 64, v);
    dft64_over_a<(PRUNE & PRUNE_IN) != 0>(v, inv);
    dft64_over_b(v, inv);
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int p = 0; p < 8; ++p) x[(q + 8 * p) * kPitch64 + j] = v[8 * q + p];
    // the second stage's w, w^2, w^4 and w^8, w^16, w^32, asked for before the barrier
    const float4 *row = reinterpret_cast<const float4 *>(bases) + 3 * j;
    const float4 a = __ldg(row), b = __ldg(row + 1), c = __ldg(row + 2);
    const float s = inv ? -1.f : 1.f;
    const float2 w1[3] = {make_float2(a.x, s * a.y), make_float2(a.z, s * a.w), make_float2(b.x, s * b.y)};
    const float2 w8[3] = {make_float2(b.z, s * b.w), make_float2(c.x, s * c.y), make_float2(c.z, s * c.w)};
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = x[j * kPitch64 + i];
    // w^(8 a + b) = (w^8)^a w^b: the first factor before the DFTs over a, the second after
    mul_rows(v, w8);
    dft64_over_a<false>(v, inv);
    mul_rows(v, w1);
    dft64_over_b(v, inv);
    float2 o[64];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int p = 0; p < 8; ++p) o[q + 8 * p] = v[8 * q + p];
    store(std::bool_constant<(PRUNE & PRUNE_OUT) != 0>{}, t, j, 64, o);
}

// One transform of the compile-time size N by T threads: input in buf in
// natural order (see first_inplace for live; HELD as in fft_inplace), or read through load.
template <int N, int T, bool HELD, int PRUNE = 0, class Between, class Store>
__device__ __forceinline__ void fft_static_inplace(float2 *buf, bool inv, int tid, Between between, Store store,
                                                   const fftst::RowTw<N, T> &rt, uint32_t live) {
    using Rd = fftst::Radices<N>;
    static_assert((PRUNE & fftst::PRUNE_IN) == 0, "inputs already in the buffer are not pruned");
    static_assert(T == N / Rd::r0, "one first-stage butterfly per thread");
    fftst::first_inplace<N>(buf, inv, tid, live);
    fftst::later<N, 1, T, Rd::r1, Rd::r0, false, 0>(buf, nullptr, inv, tid, rt.s2, store);
    if constexpr (HELD)
        fftst::last_held<N, T, Rd::r2, Rd::r0 * Rd::r1, PRUNE>(buf, tid, inv, rt.s3, between, store);
    else
        fftst::later<N, 1, T, Rd::r2, Rd::r0 * Rd::r1, true, PRUNE>(buf, nullptr, inv, tid, rt.s3, store);
}
template <int N, int T, int PRUNE = 0, class Load, class Store>
__device__ __forceinline__ void fft_static_row(float2 *buf, bool inv, int tid, Load load, Store store,
                                               const fftst::RowTw<N, T> &rt) {
    using Rd = fftst::Radices<N>;
    fftst::first<N, 1, T, PRUNE>(buf, inv, tid, load);
    fftst::later<N, 1, T, Rd::r1, Rd::r0, false, 0>(buf, nullptr, inv, tid, rt.s2, store);
    fftst::later<N, 1, T, Rd::r2, Rd::r0 * Rd::r1, true, PRUNE>(buf, nullptr, inv, tid, rt.s3, store);
}

// COUNT transforms of the compile-time size N by T threads (see fft_many for the contract).
template <int N, int COUNT, int T, int PRUNE = 0, class Load, class Store>
__device__ __forceinline__ void fft_static(float2 *buf, const float2 *__restrict__ tw, bool inv, int tid, Load load,
                                           Store store) {
    using Rd = fftst::Radices<N>;
    fftst::first<N, COUNT, T, PRUNE>(buf, inv, tid, load);
    fftst::later<N, COUNT, T, Rd::r1, Rd::r0, false, 0>(buf, tw, inv, tid, fftst::NoTw{}, store);
    fftst::later<N, COUNT, T, Rd::r2, Rd::r0 * Rd::r1, true, PRUNE>(buf, tw, inv, tid, fftst::NoTw{}, store);
}

}  // namespace ws
