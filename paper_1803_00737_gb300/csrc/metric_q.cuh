// Wang-Bovik Q of one 32 x 32 window from exact integer sums, shared by the
// metric passes (metrics.cu) and the fused forward + metrics kernel
// (fuse_metrics.cu).  The quality index (Sec. 4 / Table 3 report QNR without
// defining it):  Q = 4 s_xy mu_x mu_y / ((s_x^2 + s_y^2)(mu_x^2 + mu_y^2)).
#pragma once

#include <cstdint>

namespace dwtfuse {

constexpr int kQWinPx = 32 * 32;  // pixels per window

// Position of band pair (b, c), b < c < nb, among the pair sums (b-major
// order); the band-PAN pairs follow at nb(nb-1)/2 + b.  Loops over pairs run
// b and c over [0, nb) with a `c > b` test, so that both have constant trip
// counts, unroll fully, and the position is a compile-time constant (a
// triangular inner loop stays a loop and its sums go to local memory).
__host__ __device__ constexpr int pair_index(int nb, int b, int c) { return b * nb - b * (b + 1) / 2 + (c - b - 1); }

// Q of one window, given exact integer sums (8-bit data).  ys = scale of y.
__device__ __forceinline__ float q_exact(long long sx, long long sxx, long long sy, long long syy,
                                         long long sxy, int ys) {
    const long long n = kQWinPx;
    const long long vx = n * sxx - sx * sx;                 // n^2 var(x)
    const long long vy = n * syy - sy * sy;                 // ys^2 n^2 var(y)
    const long long cxy = n * sxy - sx * sy;                // ys n^2 cov(x, y)
    const long long ax = sx + 128 * n;                      // n mean(X)
    const long long ay = sy + 128 * n * ys;                 // ys n mean(Y)
    const float inv = 1.0f / (float)ys, inv2 = inv * inv;
    const float fvx = (float)vx, fvy = (float)vy * inv2, fc = (float)cxy * inv;
    const float fax = (float)ax, fay = (float)ay * inv;
    const float den = (fvx + fvy) * (fax * fax + fay * fay);
    if (vx + vy == 0 || (ax == 0 && ay == 0)) {
        // zero denominator: identical windows <=> sum (ys x - y)^2 = 0
        const long long d2 = (long long)ys * ys * sxx - 2LL * ys * sxy + syy;
        return (d2 == 0) ? 1.0f : 0.0f;
    }
    return 4.0f * fc * fax * fay / den;
}

// Sum of windows' Q values (FP32), exact: the integers hi and lo, in units of
// 2^-32 and 2^-77.  A window's Q is 0 or at least 2^-54 in size: the least is a
// y of one quarter grey level (4 PAN~ = 1 in one pixel; cov = 1/4 in units of
// n^2) against an x of mean m and the largest variance m (255 - m), which gives
// 1 / (4 n^3 m^2 (255 - m)) > 2^-53.3.  So every Q, and every FP32 sum of them,
// is a multiple of 2^-77.  Room: the largest images hold 2^30 windows (sides of
// 2^20), |hi| <= 2^62; an addend's lo is below 2^45, and a pass adds at most
// 1024 CTAs x 256 slots = 2^18 of them.  From the float's bits: conversions to
// 64 bits and FP64 adds run at a few lanes a clock and SM (a CTA's 256 slots of
// 21 pairs through three __float2ll_rn: 3 us at the end of the PAN pass).
struct QSum {
    long long hi = 0, lo = 0;
    __device__ __forceinline__ void add(float q) {
        const uint32_t w = __float_as_uint(q);
        const int s = (int)((w >> 23) & 255u) - 73;  // q = +-m * 2^(s - 77); 0 where s <= -24
        const unsigned long long m = (w & 0x7fffffu) | 0x800000u;
        long long h = 0, l = 0;
        if (s >= 45) {
            h = (long long)(m << (s - 45));
        } else if (s >= 0) {
            h = (long long)(m >> (45 - s));
            l = (long long)((m << s) & ((1ull << 45) - 1));
        } else if (s > -24) {  // below 2^-54: what windows that nearly cancel leave (whole units of 2^-77)
            l = (long long)(m >> -s);
        }
        hi += (w >> 31) ? -h : h;
        lo += (w >> 31) ? -l : l;
    }
    __device__ __forceinline__ void warp_sum() {
        for (int o = 16; o > 0; o >>= 1) {
            hi += __shfl_xor_sync(0xffffffffu, hi, o);
            lo += __shfl_xor_sync(0xffffffffu, lo, o);
        }
    }
};
__device__ __forceinline__ double q_value(long long hi, long long lo) {
    return (double)hi * 0x1p-32 + (double)lo * 0x1p-77;
}

// Columns of a CTA's partial row, 8-bit passes (int64): the P pairs' QSum::hi,
// nb sums (squared errors, MS values), the status of the bulk-copy waits, the
// P pairs' QSum::lo.
__host__ __device__ constexpr int metric_lo_column(int nb) { return nb * (nb + 1) / 2 + nb + 1; }

}  // namespace dwtfuse
