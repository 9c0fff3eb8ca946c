// Host/device description of one shared-memory FFT (see fft.cuh).
#pragma once

#ifdef __CUDACC__
#define WS_HD __host__ __device__
#else
#define WS_HD
#endif

namespace ws {

// Threads a CTA of the runtime plans may have: with two CTAs per SM they leave
// 128 registers per thread, enough for a radix-28 butterfly (56 values).
constexpr int kMaxFftThreads = 256;
constexpr int kMaxFftStages = 6;

// Element e of a transform sits at shared-memory slot e + e / chunk.  chunk is a
// product of leading radices, so a butterfly's elements (L apart) are `step`
// slots apart whatever its position.
struct FftPlan {
    int n;                          // transform length
    int nstages;
    int radix[kMaxFftStages];       // stage radices, first stage first
    int L[kMaxFftStages];           // radix[0] * ... * radix[s-1]
    int nb[kMaxFftStages];          // butterflies of stage s: n / radix[s]
    int twstep[kMaxFftStages];      // n / (radix[s] L[s])
    int bases[kMaxFftStages];       // the stage's twiddle bases in the twiddle buffer (fft_tables)
    int step[kMaxFftStages];        // slots from one element of a butterfly to the next
    int fuse[kMaxFftStages];        // 1: this stage and the next run as one pass (rows of forward plans)
    int slots;                      // the first stage's output slots, as integers in the twiddle buffer (fft_tables)
    // div_mul of L[s] and of chunk.
    // x / d = umulhi(x, mul) exactly for 0 <= x < 2^16 and d < 2^13, since
    // x (mul d - 2^32) < 2^32 (div_small in fft.cuh)
    unsigned L_mul[kMaxFftStages], chunk_mul;
    int stride;                     // float2 slots per transform buffer (== 8 mod 16)
    int row_threads, col_threads;   // threads per CTA: one transform (rows), two (columns)
    int box_blocks, boxes;          // TMA row copies: boxes of box_blocks column blocks
};

// Powers of a butterfly's twiddle w that a later stage's table holds (in a row of that many
// pairs); the other powers are products of these.  Forward: w, and w^4 from radix 8 on, as
// ever, which keeps the model visibilities' last bits.  Inverse: w, w^2 and, above radix 4,
// w^4 and w^8: the inverse plans have radices 6, 12, 16 or 20 where the forward ones have 3s and
// 8s, and with w and w^4 alone (w alone at radix 6) their powers' rounding moved the error
// against the exact DFT: N' = 4320 (20 6 6 6) 1.96e-7 -> 2.50e-7, 1536 (16 16 6)
// 1.97e-7 -> 2.21e-7, 3072 (16 16 12) 2.08e-7 -> 2.27e-7.
WS_HD constexpr int base_row(int radix, bool inverse) {
    return inverse ? (radix > 4 ? 4 : 2) : (radix >= 8 ? 2 : 1);
}

// ceil(2^32 / d), or 0 for d = 1
WS_HD constexpr unsigned div_mul(int d) {
    return d <= 1 ? 0u : (unsigned)((4294967296ull + (unsigned long long)d - 1ull) / (unsigned long long)d);
}

}  // namespace ws
