// Register-resident small DFTs of two transforms at once (adjacent antennas of the F-engine, adjacent
// image columns of the 256 x 256 imaging kernels), as packed FP32 pairs.
#pragma once
#include "dft.cuh"

namespace epic {

// Two complex values as packed FP32 pairs, re = (re_0, re_1) and im = (im_0, im_1), so that one f32x2
// instruction does an operation for both and the address arithmetic and twiddle loads of a thread serve both.
struct P2 { unsigned long long re, im; };

// (a - b) * exp(SIGN 2 pi i m / M) for a compile-time rotation; the half and quarter turns cost
// no multiplies (the swap and the sign go into the subtraction).
template <int SIGN>
__device__ __forceinline__ P2 sub_rot(const P2& a, const P2& b, int m, int M) {
    const int r = ((m % M) + M) % M;
    P2 d;
    if (r == 0) {
        d.re = f2sub(a.re, b.re);
        d.im = f2sub(a.im, b.im);
    } else if (2 * r == M) {
        d.re = f2sub(b.re, a.re);
        d.im = f2sub(b.im, a.im);
    } else if (4 * r == M || 4 * r == 3 * M) {
        if ((SIGN > 0) == (4 * r == M)) {      // times +i: (-(a - b).im, (a - b).re)
            d.re = f2sub(b.im, a.im);
            d.im = f2sub(a.re, b.re);
        } else {                               // times -i: ((a - b).im, -(a - b).re)
            d.re = f2sub(a.im, b.im);
            d.im = f2sub(b.re, a.re);
        }
    } else {
        const int idx = r * (64 / M);
        const float c = kTw64.c[idx], s = SIGN > 0 ? kTw64.s[idx] : -kTw64.s[idx];
        const unsigned long long dre = f2sub(a.re, b.re), dim = f2sub(a.im, b.im);
        d.re = f2fma(dre, f2dup(c), f2mul(dim, f2dup(-s)));
        d.im = f2fma(dre, f2dup(s), f2mul(dim, f2dup(c)));
    }
    return d;
}

// In-place x[k] <- sum_n x[n] exp(SIGN 2 pi i n k / N) for both values of every pair, N a power
// of two <= 64: radix-2 decimation in frequency, then a compile-time permutation.
template <int N, int SIGN>
__device__ __forceinline__ void dft2(P2 (&x)[N]) {
    if constexpr (N > 1) {
#pragma unroll
        for (int half = N / 2; half >= 1; half >>= 1) {
#pragma unroll
            for (int blk = 0; blk < N; blk += 2 * half) {
#pragma unroll
                for (int j = 0; j < half; ++j) {
                    const P2 a = x[blk + j], b = x[blk + j + half];
                    x[blk + j].re = f2add(a.re, b.re);
                    x[blk + j].im = f2add(a.im, b.im);
                    x[blk + j + half] = sub_rot<SIGN>(a, b, j, 2 * half);
                }
            }
        }
        P2 y[N];
#pragma unroll
        for (int k = 0; k < N; ++k) y[k] = x[bitrev<N>(k)];
#pragma unroll
        for (int k = 0; k < N; ++k) x[k] = y[k];
    }
}

}  // namespace epic
