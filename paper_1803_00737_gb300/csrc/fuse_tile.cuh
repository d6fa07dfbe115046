// Warp-strip tile machinery of the fused DWT pansharpening forward pass.
//
// Method (arXiv:1803.00737 Sec. 2): F_b = IDWT2(DWT2(P) with LL <- gain * M_b).
// The map is linear, so with L the low-pass half of the analysis matrix and U
// the synthesis of an LL-only coefficient image,
//     F_b = P + U(E_b),   E_b = gain * M_b - LL(P),   LL(P) = L_H P L_W^T.
// The detail subbands (HL, LH, HH) are never formed: they pass through
// unchanged, and the identity above is what remains of them.  LL(P) is
// computed once per tile and reused for every band.
//
//  Haar (Eq. 1-2, 11-12):  LL(i,j) = mean of the 2x2 block (i,j)  (rows, then
//                          columns, as the paper orders them), U = repeat 2x2.
//  D4   (Eq. 3-8, 13-16):  LL(i,j) = sum_{a,b} h_a h_b P(2i+a, 2j+b)   (mod H, W)
//                          U(E)(2m+r, 2n+q) = sum_{a,b in 0,1} h_{r+2a} h_{q+2b} E(m-a, n-b)
//
// Work unit: one warp owns a strip of 128 PAN columns (4 per lane: x..x+3,
// MS columns n = x/2 and n+1) and walks down R MS rows.  Everything stays in
// registers: D4 needs, per lane and PAN row, the 8 PAN columns x-2..x+5
// (periodic wrap at the image edges, Eq. 5-6 and 13-14), and a vertical
// pipeline keeps the row-synthesised values of MS row m-1 for row m.  Loads
// use the read-only path; fused rows are written with streaming stores.
//
// What bounds the walkers: with a float output HBM writes; with only the uint8
// product, or scoring it, the instructions per pixel and the latency of a
// step's loads (16 warps per SM).  So: paired FP32, byte conversions on the
// fast pipes, running addresses instead of 64-bit products per band, row
// layouts and inner strips (no wrapped columns) as template instances.  Per
// warp step of 8 bands 1000 -> 585 instructions; against the walkers with
// run-time layouts and scalar FP32: 7480 x 8140 x 8 to uint8 279 -> 185 us,
// scored 9414^2 x 8 1022 -> 894 us and 16384^2 x 6 1624 -> 1589 us a pass.
// Streaming the rows through a per-warp cp.async ring instead of registers
// (615 instructions per step) was slower: 7480 x 8140 x 8 237 us, 16384^2 x 6
// scored 1831 us.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace dwtfuse {

constexpr int kWarpCols = 128;  // PAN columns per warp strip
constexpr int kMaxBands = 16;

// Daubechies-4 low-pass h of Eq. 7-8: (1+sqrt3, 3+sqrt3, 3-sqrt3, 1-sqrt3) / (4 sqrt2).
constexpr float kH0 = 0.48296291314453414f;
constexpr float kH1 = 0.83651630373780794f;
constexpr float kH2 = 0.22414386804201339f;
constexpr float kH3 = -0.12940952255126037f;

// ------------------------------------------------------------------ scalar helpers

// Exact uint8 -> float: place the byte in the mantissa of 2^23 and subtract.
__device__ __forceinline__ float byte_f(uint32_t word, int k) {
    return __int_as_float(__byte_perm(word, 0x4B000000u, 0x7440u | (uint32_t)k)) - 8388608.0f;
}

// float -> uint8: clamp to [0, 255], round half to even (cvt saturates).
__device__ __forceinline__ uint32_t f2u8(float v) {
    uint32_t r;
    asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ uint32_t pack4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040u), __byte_perm(c, d, 0x0040u), 0x5410u);
}

__device__ __forceinline__ int64_t wrap(int64_t i, int64_t n) {
    return i < 0 ? i + n : (i >= n ? i - n : i);
}

// ------------------------------------------------------------------ loads

// Two consecutive pixels starting at an even column (always in bounds).
__device__ __forceinline__ void ld2(const uint8_t *p, float &a, float &b) {
    const uint32_t w = __ldg(reinterpret_cast<const unsigned short *>(p));
    a = byte_f(w, 0);
    b = byte_f(w, 1);
}
__device__ __forceinline__ void ld2(const float *p, float &a, float &b) {
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    a = v.x;
    b = v.y;
}
// Four consecutive pixels starting at a column that is a multiple of 4 (aligned path).
__device__ __forceinline__ void ld4(const uint8_t *p, float *v) {
    const uint32_t w = __ldg(reinterpret_cast<const unsigned int *>(p));
    v[0] = byte_f(w, 0);
    v[1] = byte_f(w, 1);
    v[2] = byte_f(w, 2);
    v[3] = byte_f(w, 3);
}
__device__ __forceinline__ void ld4(const float *p, float *v) {
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}

// ------------------------------------------------------------------ stores

struct OutPtrs {
    float *f32;   // band plane base or nullptr
    uint8_t *u8;  // band plane base or nullptr
};

// Writes the 4 fused pixels (y, x..x+3) of one band.  `two` = x+2 < W.
__device__ __forceinline__ void store4(const OutPtrs &o, int64_t off, bool a4, bool two,
                                       const float *v) {
    if (o.f32) {
        float *p = o.f32 + off;
        if (a4) {
            __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
        } else {
            __stcs(reinterpret_cast<float2 *>(p), make_float2(v[0], v[1]));
            if (two) __stcs(reinterpret_cast<float2 *>(p + 2), make_float2(v[2], v[3]));
        }
    }
    if (o.u8) {
        const uint32_t q0 = f2u8(v[0]), q1 = f2u8(v[1]), q2 = f2u8(v[2]), q3 = f2u8(v[3]);
        uint8_t *p = o.u8 + off;
        if (a4) {
            __stcs(reinterpret_cast<unsigned int *>(p), pack4(q0, q1, q2, q3));
        } else {
            __stcs(reinterpret_cast<unsigned short *>(p), (unsigned short)(q0 | (q1 << 8)));
            if (two) __stcs(reinterpret_cast<unsigned short *>(p + 2), (unsigned short)(q2 | (q3 << 8)));
        }
    }
}

// ------------------------------------------------------------------ scene

// Everything a warp needs about one scene.  Band pointers are typed by the
// kernel template (TIn); the plane stride of the outputs is out_plane.
struct SceneArgs {
    const void *pan;
    const void *ms[kMaxBands];
    float *out_f32;
    uint8_t *out_u8;
    int64_t H, W;
    int32_t bands;
    int32_t wavelet;   // 0 Haar, 1 D4
    int32_t in_f32;    // inputs are float (else uint8)
    float gain;
    int32_t a4;        // W % 4 == 0 and PAN/outputs aligned for 4-pixel vectors
    int32_t alt;       // W % 4 == 2 with aligned planes: even rows aligned, odd rows 2 px past
    int64_t out_plane; // elements between output band planes (H * W for a whole scene)
    int32_t m_lo;      // MS rows [m_lo, m_hi) are fused; output row 0 belongs to MS row m_lo
    int32_t m_hi;      // (0 and H/2 for a whole scene; a row band's slab starts past its halo)
};

// Column bookkeeping of one lane for one strip (sides are < 2^20, so 32 bits).
struct LaneCols {
    int32_t x;           // first PAN column (even); clamped to 0 for idle lanes
    int32_t cm, c2, c4;  // wrapped starts of the pixel pairs x-2, x+2, x+4
    int32_t nA, nB, nC;  // MS columns n-1 (wrapped), n, n+1 (wrapped)
    bool active;         // x < W
    bool two;            // x + 2 < W (second MS column exists)
    bool last;           // last active lane of the strip (x + 4 >= W or lane 31)
};

__device__ __forceinline__ int32_t wrap32(int32_t i, int32_t n) {
    return i < 0 ? i + n : (i >= n ? i - n : i);
}

__device__ __forceinline__ LaneCols lane_cols(int64_t x0, int lane, int64_t W64) {
    LaneCols c;
    const int32_t W = (int32_t)W64;
    int32_t x = (int32_t)x0 + 4 * lane;
    c.active = x < W;
    if (!c.active) x = 0;
    c.x = x;
    c.two = x + 2 < W;
    c.last = lane == 31 || x + 4 >= W;
    c.cm = wrap32(x - 2, W);
    c.c2 = wrap32(x + 2, W);
    c.c4 = wrap32(x + 4, W);
    c.c4 = c.c4 >= W ? c.c4 - W : c.c4;
    const int32_t W2 = W >> 1, n = x >> 1;
    c.nA = wrap32(n - 1, W2);
    c.nB = n;
    c.nC = wrap32(n + 1, W2);
    return c;
}

// PAN row y: the 8 pixels x-2..x+5 (D4) with periodic wrap.
template <typename T>
__device__ __forceinline__ void load_row8(const T *row, const LaneCols &c, bool a4, float *v) {
    ld2(row + c.cm, v[0], v[1]);
    if (a4) {
        ld4(row + c.x, v + 2);
    } else {
        ld2(row + c.x, v[2], v[3]);
        ld2(row + c.c2, v[4], v[5]);
    }
    ld2(row + c.c4, v[6], v[7]);
}

// PAN row y: the 4 pixels x..x+3 (Haar; columns past W read column 0, unused).
template <typename T>
__device__ __forceinline__ void load_row4(const T *row, const LaneCols &c, bool a4, float *v) {
    if (a4) {
        ld4(row + c.x, v);
    } else {
        ld2(row + c.x, v[0], v[1]);
        ld2(row + c.c2, v[2], v[3]);
    }
}

// D4 row low-pass R(y, n') = sum_b h_b P(y, 2n'+b) for n' = n-1, n, n+1.
__device__ __forceinline__ void d4_rowpass(const float *v, float *r) {
    r[0] = fmaf(kH3, v[3], fmaf(kH2, v[2], fmaf(kH1, v[1], kH0 * v[0])));
    r[1] = fmaf(kH3, v[5], fmaf(kH2, v[4], fmaf(kH1, v[3], kH0 * v[2])));
    r[2] = fmaf(kH3, v[7], fmaf(kH2, v[6], fmaf(kH1, v[5], kH0 * v[4])));
}

// ------------------------------------------------------------------ row layouts
//
// kVec:   W % 4 == 0 and every image row starts on a 4-pixel boundary.
// kShift: W % 4 == 2 with aligned planes: even rows start on a 4-pixel
//         boundary, odd rows 2 pixels past one.
// kPairs: anything else (every access is a pixel pair).
enum : int { kPairs = 0, kVec = 1, kShift = 2 };

__device__ __host__ inline int row_layout(int32_t a4, int32_t alt) { return a4 ? kVec : (alt ? kShift : kPairs); }

// A strip is inner when no lane's taps (columns x-2 .. x+5, MS columns
// n-1 .. n+1) leave the image row: the wrapped columns are then plain offsets
// and every lane is active.  The same for the whole warp.
__device__ __forceinline__ bool strip_inner(int64_t x0, int64_t W) { return x0 > 0 && x0 + kWarpCols + 2 <= W; }

// ------------------------------------------------------------------ paired FP32
//
// Two FP32 operations per instruction (fma / mul / add .f32x2, each lane
// rounded as the scalar operation): the same arithmetic pipe time, half the
// issue slots.  The forward walkers were issue-bound (uint8 output, 8 bands:
// 74 % of issue slots, about 1000 instructions per warp and MS row).
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pk2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void up2(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// 4 floats -> 4 uint8 (clamped, rounded half to even; NaN -> 0) in one word.
// cvt.rni.s32 saturates, and cvt.pack clamps two values to bytes at once: 6
// instructions against 4 saturating conversions and 3 byte permutes.
__device__ __forceinline__ uint32_t pack4u8(const float *v) {
    int i0, i1, i2, i3;
    asm("cvt.rni.s32.f32 %0, %1;" : "=r"(i0) : "f"(v[0]));
    asm("cvt.rni.s32.f32 %0, %1;" : "=r"(i1) : "f"(v[1]));
    asm("cvt.rni.s32.f32 %0, %1;" : "=r"(i2) : "f"(v[2]));
    asm("cvt.rni.s32.f32 %0, %1;" : "=r"(i3) : "f"(v[3]));
    uint32_t hi, w;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(i3), "r"(i2));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(w) : "r"(i1), "r"(i0), "r"(hi));
    return w;
}

// ------------------------------------------------------------------ raw loads
//
// A walker's inputs as loaded: uint8 words and bytes (a third of the floats'
// registers), converted where they are used.

template <typename T>
struct RawRow;  // PAN columns x-2 .. x+5 of one image row
template <>
struct RawRow<uint8_t> {
    uint32_t a, b, c, d;
};
template <>
struct RawRow<float> {
    float v[8];
};

// W8: all 8 columns (D4); else columns x .. x+3 only (Haar).  SHIFT: the row
// starts 2 pixels past a 4-pixel boundary (kShift, odd rows).
template <int LAY, bool INNER, bool SHIFT, bool W8>
__device__ __forceinline__ void load_raw(const uint8_t *row, const LaneCols &c, RawRow<uint8_t> &r) {
    if (LAY == kVec) {
        r.b = __ldg(reinterpret_cast<const unsigned int *>(row + c.x));
        if (W8) {
            if (INNER) {
                r.a = __ldg(reinterpret_cast<const unsigned short *>(row + c.x - 2));
                r.c = __ldg(reinterpret_cast<const unsigned short *>(row + c.x + 4));
            } else {
                r.a = __ldg(reinterpret_cast<const unsigned short *>(row + c.cm));
                r.c = __ldg(reinterpret_cast<const unsigned short *>(row + c.c4));
            }
        }
        return;
    }
    if (LAY == kShift && INNER) {
        const uint8_t *p = row + c.x;
        if (SHIFT) {
            if (W8) {
                r.a = __ldg(reinterpret_cast<const unsigned int *>(p - 2));
                r.b = __ldg(reinterpret_cast<const unsigned int *>(p + 2));
            } else {
                r.a = __ldg(reinterpret_cast<const unsigned short *>(p));
                r.b = __ldg(reinterpret_cast<const unsigned short *>(p + 2));
            }
        } else {
            r.b = __ldg(reinterpret_cast<const unsigned int *>(p));
            if (W8) {
                r.a = __ldg(reinterpret_cast<const unsigned short *>(p - 2));
                r.c = __ldg(reinterpret_cast<const unsigned short *>(p + 4));
            }
        }
        return;
    }
    if (W8) {
        r.a = __ldg(reinterpret_cast<const unsigned short *>(row + c.cm));
        r.d = __ldg(reinterpret_cast<const unsigned short *>(row + c.c4));
    }
    r.b = __ldg(reinterpret_cast<const unsigned short *>(row + c.x));
    r.c = __ldg(reinterpret_cast<const unsigned short *>(row + c.c2));
}

template <int LAY, bool INNER, bool SHIFT, bool W8>
__device__ __forceinline__ void load_raw(const float *row, const LaneCols &c, RawRow<float> &r) {
    if (LAY == kVec || (LAY == kShift && INNER)) {
        const float *p = row + c.x;
        if (LAY == kShift && SHIFT) {
            if (W8) {
                ld4(p - 2, r.v);
                ld4(p + 2, r.v + 4);
            } else {
                ld2(p, r.v[2], r.v[3]);
                ld2(p + 2, r.v[4], r.v[5]);
            }
            return;
        }
        ld4(p, r.v + 2);
        if (W8) {
            if (LAY == kShift || INNER) {
                ld2(p - 2, r.v[0], r.v[1]);
                ld2(p + 4, r.v[6], r.v[7]);
            } else {
                ld2(row + c.cm, r.v[0], r.v[1]);
                ld2(row + c.c4, r.v[6], r.v[7]);
            }
        }
        return;
    }
    ld2(row + c.x, r.v[2], r.v[3]);
    ld2(row + c.c2, r.v[4], r.v[5]);
    if (W8) {
        ld2(row + c.cm, r.v[0], r.v[1]);
        ld2(row + c.c4, r.v[6], r.v[7]);
    }
}

// The row's words: lo = columns x-2 .. x+1, hi = x+2 .. x+5 (Haar: only the
// own columns x .. x+3, in lo).
template <int LAY, bool INNER, bool SHIFT, bool W8>
__device__ __forceinline__ void raw_words(const RawRow<uint8_t> &r, uint32_t &lo, uint32_t &hi) {
    if (LAY == kVec || (LAY == kShift && INNER && !SHIFT)) {
        if (W8) {
            lo = __byte_perm(r.a, r.b, 0x5410u);
            hi = __byte_perm(r.b, r.c, 0x5432u);
        } else {
            lo = r.b;
        }
    } else if (LAY == kShift && INNER) {
        if (W8) {
            lo = r.a;
            hi = r.b;
        } else {
            lo = __byte_perm(r.a, r.b, 0x5410u);
        }
    } else if (W8) {
        lo = __byte_perm(r.a, r.b, 0x5410u);
        hi = __byte_perm(r.c, r.d, 0x5410u);
    } else {
        lo = __byte_perm(r.b, r.c, 0x5410u);
    }
}

// Columns x-2 .. x+5 (D4: v[0..7]; Haar: only v[2..5]) as floats, and the own
// columns' word x .. x+3 (uint8 only).
template <int LAY, bool INNER, bool SHIFT, bool W8>
__device__ __forceinline__ void raw_floats(const RawRow<uint8_t> &r, float *v, uint32_t &own) {
    uint32_t lo, hi = 0;
    raw_words<LAY, INNER, SHIFT, W8>(r, lo, hi);
    if (W8) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = byte_f(lo, k);
            v[4 + k] = byte_f(hi, k);
        }
        own = __byte_perm(lo, hi, 0x5432u);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[2 + k] = byte_f(lo, k);
        own = lo;
    }
}
template <int LAY, bool INNER, bool SHIFT, bool W8>
__device__ __forceinline__ void raw_floats(const RawRow<float> &r, float *v, uint32_t &own) {
#pragma unroll
    for (int k = W8 ? 0 : 2; k < (W8 ? 8 : 6); ++k) v[k] = r.v[k];
    own = 0;
}

// One MS value, raw and as a float.  uint8: the byte in a 32-bit register
// (cvt.rn.f32.u32 runs at 64 lanes a clock and SM, cvt.rn.f32.u8 at 16).
template <typename T>
struct RawMs;
template <>
struct RawMs<uint8_t> {
    typedef uint32_t type;
};
template <>
struct RawMs<float> {
    typedef float type;
};
__device__ __forceinline__ uint32_t ld_ms(const uint8_t *p) {
    uint32_t r;
    asm("ld.global.nc.u8 %0, [%1];" : "=r"(r) : "l"(p));
    return r;
}
__device__ __forceinline__ float ld_ms(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ms_f(uint32_t v) {
    float f;
    asm("cvt.rn.f32.u32 %0, %1;" : "=f"(f) : "r"(v));
    return f;
}
__device__ __forceinline__ float ms_f(float v) { return v; }

// ------------------------------------------------------------------ row walkers
//
// A walker takes one lane's columns (LaneCols) down MS rows [m_s, m_e) and
// hands every band's two fused PAN rows 2m, 2m+1 (4 pixels per lane) to an
// emitter: out.band(b, v0, v1, mn, mn1) per band, with the band's raw MS
// values at MS columns n = x/2 and n+1 (the ones the lane's pixels were made
// from), then out.row_end(m, own0, own1) once per MS row with the lane's PAN
// words of rows 2m and 2m+1 (uint8 images).  Emit::kAllLanes: the emitter
// needs every lane (warp shuffles, barriers), so idle lanes compute on column
// 0 and call it too.  Addresses run: one PAN pointer and one MS offset are
// advanced per MS row.

// Emit::kMode, a sum of:
//   kAheadPan, kAheadMs  load the next MS row's PAN rows / MS values one row
//                        ahead (raw words and bytes; they stay in registers
//                        for a whole row)
//   kScalarCol, kScalarRow  column / row synthesis in scalar FP32 (its
//                        constants are immediates; the paired form holds 8 and
//                        4 registers of them)
// Chosen per kernel by measurement (see there): loads ahead pay where few bands
// leave registers free, paired FP32 where instructions bound the kernel and
// nothing spills.
enum : int { kAheadPan = 1, kAheadMs = 2, kScalarCol = 4, kScalarRow = 8 };

// Haar (Eq. 1-2, 11-12).
template <typename T, int NB, int LAY, bool INNER, class Emit>
__device__ __forceinline__ void haar_rows(const SceneArgs &s, const LaneCols &c, int m_s, int m_e,
                                          int b0, Emit &out) {
    typedef typename RawMs<T>::type M;
    constexpr bool kPanA = (Emit::kMode & kAheadPan) != 0, kMsA = (Emit::kMode & kAheadMs) != 0;
    const int64_t W = s.W, W2 = W >> 1;
    const T *pan = static_cast<const T *>(s.pan) + (int64_t)(2 * m_s) * W;
    int64_t mo = (int64_t)m_s * W2 + c.nB;
    const int dC = c.nC - c.nB;
    RawRow<T> ra, rb;
    M mr[NB][2];
    auto load_pan = [&]() {
        load_raw<LAY, INNER, false, false>(pan, c, ra);
        load_raw<LAY, INNER, true, false>(pan + W, c, rb);
        pan += 2 * W;
    };
    auto load_ms = [&](int b) {
        const T *ms = static_cast<const T *>(s.ms[b0 + b]) + mo;
        mr[b][0] = ld_ms(ms);
        mr[b][1] = INNER ? ld_ms(ms + 1) : ld_ms(ms + dC);
    };
    if (kPanA) load_pan();
    if (kMsA) {
#pragma unroll
        for (int b = 0; b < NB; ++b) load_ms(b);
    }
#pragma unroll 1
    for (int m = m_s; m < m_e; ++m) {
        const bool more = m + 1 < m_e;
        if (!kPanA) load_pan();
        if (!kMsA) {
#pragma unroll
            for (int b = 0; b < NB; ++b) load_ms(b);
        }
        mo += W2;
        float p0[8], p1[8];
        uint32_t own0, own1;
        raw_floats<LAY, INNER, false, false>(ra, p0, own0);
        raw_floats<LAY, INNER, true, false>(rb, p1, own1);
        if (kPanA && more) load_pan();
        // Eq. 1 along the rows, then along the columns: LL = 2x2 mean (exact in FP32 for 8-bit input).
        const float ll0 = ((p0[2] + p0[3]) * 0.5f + (p1[2] + p1[3]) * 0.5f) * 0.5f;
        const float ll1 = ((p0[4] + p0[5]) * 0.5f + (p1[4] + p1[5]) * 0.5f) * 0.5f;
        const f32x2 pa0 = pk2(p0[2], p0[3]), pa1 = pk2(p0[4], p0[5]);
        const f32x2 pb0 = pk2(p1[2], p1[3]), pb1 = pk2(p1[4], p1[5]);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            // Eq. 11-12 on an LL-only image repeat each coefficient over its 2x2 block.
            const M m0 = mr[b][0], m1 = mr[b][1];
            if (kMsA && more) load_ms(b);  // the next row's, once this row's are taken
            const float e0 = fmaf(s.gain, ms_f(m0), -ll0);
            const float e1 = fmaf(s.gain, ms_f(m1), -ll1);
            const f32x2 ee0 = pk2(e0, e0), ee1 = pk2(e1, e1);
            float v[4], w[4];
            up2(add2(pa0, ee0), v[0], v[1]);
            up2(add2(pa1, ee1), v[2], v[3]);
            up2(add2(pb0, ee0), w[0], w[1]);
            up2(add2(pb1, ee1), w[2], w[3]);
            out.band(b, v, w, m0, m1);
        }
        out.template row_end<NB>(m, own0, own1);
    }
}

// D4 (Eq. 3-10, 13-16).
template <typename T, int NB, int LAY, bool INNER, class Emit>
__device__ __forceinline__ void d4_rows(const SceneArgs &s, const LaneCols &c, int m_s, int m_e, int b0,
                                        Emit &out) {
    typedef typename RawMs<T>::type M;
    constexpr bool kPanA = (Emit::kMode & kAheadPan) != 0, kMsA = (Emit::kMode & kAheadMs) != 0;
    const int64_t W = s.W, H = s.H, W2 = W >> 1;
    const int H2 = (int)(H >> 1);
    const T *const img = static_cast<const T *>(s.pan);
    const float gain = s.gain;
    const f32x2 h01 = pk2(kH0, kH1), h23 = pk2(kH2, kH3);
    const f32x2 h00 = pk2(kH0, kH0), h11 = pk2(kH1, kH1), h22 = pk2(kH2, kH2), h33 = pk2(kH3, kH3);
    const int dA = c.nA - c.nB, dC = c.nC - c.nB;

    // Row synthesis (Eq. 15-16 on an LL-only row, wrap of Eq. 13-14 via nA) of
    // E_b at PAN columns x .. x+3, as the pairs (x, x+1) and (x+2, x+3).
    auto synth = [&](const M *mv, const float *ll, f32x2 &lo, f32x2 &hi) {
        const float eA = fmaf(gain, ms_f(mv[0]), -ll[0]);
        const float eB = fmaf(gain, ms_f(mv[1]), -ll[1]);
        const float eC = fmaf(gain, ms_f(mv[2]), -ll[2]);
        if constexpr ((Emit::kMode & kScalarRow) != 0) {
            lo = pk2(fmaf(kH2, eA, kH0 * eB), fmaf(kH3, eA, kH1 * eB));
            hi = pk2(fmaf(kH2, eB, kH0 * eC), fmaf(kH3, eB, kH1 * eC));
            return;
        }
        const f32x2 bb = pk2(eB, eB);
        lo = fma2(h23, pk2(eA, eA), mul2(h01, bb));
        hi = fma2(h23, bb, mul2(h01, pk2(eC, eC)));
    };
    M mr[NB][3];
    auto load_ms = [&](int b, int64_t mo) {
        const T *ms = static_cast<const T *>(s.ms[b0 + b]) + mo;
        mr[b][0] = INNER ? ld_ms(ms - 1) : ld_ms(ms + dA);
        mr[b][1] = ld_ms(ms);
        mr[b][2] = INNER ? ld_ms(ms + 1) : ld_ms(ms + dC);
    };

    // Prologue: MS row mp = m_s - 1 (periodic) needs PAN rows 2mp .. 2mp+3.
    const int mp = m_s > 0 ? m_s - 1 : H2 - 1;
    float r0[3], r1[3], r2[3], r3[3];
    f32x2 pc[2], pd[2];  // own PAN pixels of rows 2m, 2m+1 for the current m
    uint32_t own0, own1;
    f32x2 hprev[NB][2];  // row synthesis of E_b(m-1, .) at PAN columns x .. x+3
    RawRow<T> ra, rb;
    {
        RawRow<T> q0, q1;
        const T *p = img + (int64_t)(2 * mp) * W;
        load_raw<LAY, INNER, false, true>(p, c, q0);
        load_raw<LAY, INNER, true, true>(p + W, c, q1);
        p = img + (int64_t)(2 * m_s) * W;
        load_raw<LAY, INNER, false, true>(p, c, ra);
        load_raw<LAY, INNER, true, true>(p + W, c, rb);
#pragma unroll
        for (int b = 0; b < NB; ++b) load_ms(b, (int64_t)mp * W2 + c.nB);
        float v[8];
        raw_floats<LAY, INNER, false, true>(q0, v, own0);
        d4_rowpass(v, r0);
        raw_floats<LAY, INNER, true, true>(q1, v, own0);
        d4_rowpass(v, r1);
        raw_floats<LAY, INNER, false, true>(ra, v, own0);
        d4_rowpass(v, r2);
        pc[0] = pk2(v[2], v[3]);
        pc[1] = pk2(v[4], v[5]);
        raw_floats<LAY, INNER, true, true>(rb, v, own1);
        d4_rowpass(v, r3);
        pd[0] = pk2(v[2], v[3]);
        pd[1] = pk2(v[4], v[5]);
        float ll[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            ll[k] = fmaf(kH3, r3[k], fmaf(kH2, r2[k], fmaf(kH1, r1[k], kH0 * r0[k])));
#pragma unroll
        for (int b = 0; b < NB; ++b) synth(mr[b], ll, hprev[b][0], hprev[b][1]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) { r0[k] = r2[k]; r1[k] = r3[k]; }

    // PAN rows 2m+2, 2m+3 (periodic: past the last row comes row 0).
    const T *pan = img + (int64_t)(m_s + 1 < H2 ? 2 * m_s + 2 : 0) * W;
    int64_t mo = (int64_t)m_s * W2 + c.nB;
    auto load_pan = [&](int m) {  // the PAN rows MS row m adds
        load_raw<LAY, INNER, false, true>(pan, c, ra);
        load_raw<LAY, INNER, true, true>(pan + W, c, rb);
        pan = m + 2 == H2 ? img : pan + 2 * W;
    };
    if (kPanA) load_pan(m_s);
    if (kMsA) {
#pragma unroll
        for (int b = 0; b < NB; ++b) load_ms(b, mo);
    }
#pragma unroll 1
    for (int m = m_s; m < m_e; ++m) {
        const bool more = m + 1 < m_e;
        if (!kPanA) load_pan(m);
        if (!kMsA) {
#pragma unroll
            for (int b = 0; b < NB; ++b) load_ms(b, mo);
        }
        mo += W2;
        float va[8], vb[8];
        uint32_t nown0, nown1;
        raw_floats<LAY, INNER, false, true>(ra, va, nown0);
        raw_floats<LAY, INNER, true, true>(rb, vb, nown1);
        if (kPanA && more) load_pan(m + 1);
        d4_rowpass(va, r2);
        d4_rowpass(vb, r3);
        float ll[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            ll[k] = fmaf(kH3, r3[k], fmaf(kH2, r2[k], fmaf(kH1, r1[k], kH0 * r0[k])));
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const M mv[3] = {mr[b][0], mr[b][1], mr[b][2]};
            if (kMsA && more) load_ms(b, mo);  // the next row's, once this row's are taken
            f32x2 hc[2];
            synth(mv, ll, hc[0], hc[1]);
            // Column synthesis: row 2m takes h0 (row m) and h2 (row m-1), row 2m+1 takes h1 and h3.
            float v0[4], v1[4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if constexpr ((Emit::kMode & kScalarCol) != 0) {
                    float g0, g1, x0, x1, c0, c1, d0, d1;
                    up2(hprev[b][q], g0, g1);
                    up2(hc[q], x0, x1);
                    up2(pc[q], c0, c1);
                    up2(pd[q], d0, d1);
                    v0[2 * q] = fmaf(kH2, g0, fmaf(kH0, x0, c0));
                    v0[2 * q + 1] = fmaf(kH2, g1, fmaf(kH0, x1, c1));
                    v1[2 * q] = fmaf(kH3, g0, fmaf(kH1, x0, d0));
                    v1[2 * q + 1] = fmaf(kH3, g1, fmaf(kH1, x1, d1));
                } else {
                    up2(fma2(h22, hprev[b][q], fma2(h00, hc[q], pc[q])), v0[2 * q], v0[2 * q + 1]);
                    up2(fma2(h33, hprev[b][q], fma2(h11, hc[q], pd[q])), v1[2 * q], v1[2 * q + 1]);
                }
                hprev[b][q] = hc[q];
            }
            out.band(b, v0, v1, mv[1], mv[2]);
        }
        out.template row_end<NB>(m, own0, own1);
#pragma unroll
        for (int k = 0; k < 3; ++k) { r0[k] = r2[k]; r1[k] = r3[k]; }
        pc[0] = pk2(va[2], va[3]);
        pc[1] = pk2(va[4], va[5]);
        pd[0] = pk2(vb[2], vb[3]);
        pd[1] = pk2(vb[4], vb[5]);
        own0 = nown0;
        own1 = nown1;
    }
}

// The walker of a wavelet over one strip: inner strips (most) run an instance
// without wrapped columns.
template <typename T, int WAV, int NB, int LAY, class Emit>
__device__ __forceinline__ void walk_rows(const SceneArgs &s, const LaneCols &c, int64_t x0, int m_s, int m_e, int b0,
                                          Emit &out) {
    if (LAY != kPairs && strip_inner(x0, s.W)) {
        if (WAV == 0)
            haar_rows<T, NB, LAY, LAY != kPairs>(s, c, m_s, m_e, b0, out);
        else
            d4_rows<T, NB, LAY, LAY != kPairs>(s, c, m_s, m_e, b0, out);
    } else {
        if (WAV == 0)
            haar_rows<T, NB, LAY, false>(s, c, m_s, m_e, b0, out);
        else
            d4_rows<T, NB, LAY, false>(s, c, m_s, m_e, b0, out);
    }
}

// ------------------------------------------------------------------ direct emitter

// Writes the lane's 4 fused pixels x .. x+3 of one band row at p (the address
// of column x).  `odd`: an odd image row; under kShift it starts 2 pixels past
// a 4-pixel boundary, and every lane but the first writes the aligned vector
// x-2 .. x+1, taking pixels x-2, x-1 from its left neighbour; lane 0 writes
// x, x+1 and the last lane of the strip (x + 4 >= W or lane 31) also
// x+2, x+3.  Under kShift every lane of the warp calls it (warp shuffles).
template <int LAY>
__device__ __forceinline__ void store_f32(float *p, const LaneCols &c, int lane, bool odd, const float *v) {
    if (LAY == kShift && odd) {
        const float p2 = __shfl_up_sync(0xffffffffu, v[2], 1);
        const float p3 = __shfl_up_sync(0xffffffffu, v[3], 1);
        if (c.active) {
            if (lane > 0)
                __stcs(reinterpret_cast<float4 *>(p - 2), make_float4(p2, p3, v[0], v[1]));
            else
                __stcs(reinterpret_cast<float2 *>(p), make_float2(v[0], v[1]));
            if (c.two && c.last) __stcs(reinterpret_cast<float2 *>(p + 2), make_float2(v[2], v[3]));
        }
        return;
    }
    if (!c.active) return;
    if (LAY == kVec || (LAY == kShift && c.two)) {
        __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
    } else {
        __stcs(reinterpret_cast<float2 *>(p), make_float2(v[0], v[1]));
        if (c.two) __stcs(reinterpret_cast<float2 *>(p + 2), make_float2(v[2], v[3]));
    }
}
// The same for the 4 rounded pixels in w.
template <int LAY>
__device__ __forceinline__ void store_u8(uint8_t *p, const LaneCols &c, int lane, bool odd, uint32_t w) {
    if (LAY == kShift && odd) {
        const uint32_t pw = __shfl_up_sync(0xffffffffu, w, 1);
        if (c.active) {
            if (lane > 0)
                __stcs(reinterpret_cast<unsigned int *>(p - 2), __byte_perm(pw, w, 0x5432u));
            else
                __stcs(reinterpret_cast<unsigned short *>(p), (unsigned short)(w & 0xffffu));
            if (c.two && c.last) __stcs(reinterpret_cast<unsigned short *>(p + 2), (unsigned short)(w >> 16));
        }
        return;
    }
    if (!c.active) return;
    if (LAY == kVec || (LAY == kShift && c.two)) {
        __stcs(reinterpret_cast<unsigned int *>(p), w);
    } else {
        __stcs(reinterpret_cast<unsigned short *>(p), (unsigned short)(w & 0xffffu));
        if (c.two) __stcs(reinterpret_cast<unsigned short *>(p + 2), (unsigned short)(w >> 16));
    }
}

// Output addresses of a lane, running: the band's fused pixels (row 2m, column
// x) of the band in hand, stepped by a plane per band and by two rows less
// the planes stepped at the end of an MS row.
struct OutRun {
    float *f;
    uint8_t *u;
    bool hf, hu;  // which outputs are wanted (the other's address is not used)
    __device__ __forceinline__ OutRun(const SceneArgs &s, const LaneCols &c, int b0, int m_s)
        : hf(s.out_f32 != nullptr), hu(s.out_u8 != nullptr) {
        const int64_t off = (int64_t)b0 * s.out_plane + (int64_t)(2 * (m_s - s.m_lo)) * s.W + c.x;
        f = s.out_f32 + off;
        u = s.out_u8 + off;
    }
    __device__ __forceinline__ void next_row(int64_t step) {
        f += step;
        u += step;
    }
};

// Every lane writes its own 4 pixels to global memory.  kVec: 4-pixel
// vectors; kShift: even rows as vectors (the lane at x = W-2 pairs), odd rows
// through the neighbour's pixels (store_f32, store_u8); kPairs: pixel pairs.
// U8ONLY: the instance for a uint8 output alone.
template <int LAY, int MODE, bool U8ONLY>
struct DirectEmit {
    static constexpr bool kAllLanes = LAY == kShift;
    static constexpr int kMode = MODE;
    const LaneCols &c;
    OutRun o;
    int64_t plane;
    int W, lane;

    __device__ __forceinline__ DirectEmit(const SceneArgs &s, const LaneCols &cc, int b0, int m_s, int ln)
        : c(cc), o(s, cc, b0, m_s), plane(s.out_plane), W((int)s.W), lane(ln) {}

    template <typename M>
    __device__ __forceinline__ void band(int, const float *v0, const float *v1, M, M) {
        if (!U8ONLY && o.hf) {
            store_f32<LAY>(o.f, c, lane, false, v0);
            store_f32<LAY>(o.f + W, c, lane, true, v1);
            o.f += plane;
        }
        if (U8ONLY || o.hu) {
            store_u8<LAY>(o.u, c, lane, false, pack4u8(v0));
            store_u8<LAY>(o.u + W, c, lane, true, pack4u8(v1));
            o.u += plane;
        }
    }
    template <int NB>
    __device__ __forceinline__ void row_end(int, uint32_t, uint32_t) {
        const int64_t step = 2 * (int64_t)W - NB * plane;
        if (!U8ONLY) o.f += step;
        o.u += step;
    }
};

// One warp strip: 128 PAN columns from x0, MS rows [m_s, m_e), bands
// [b0, b0 + NB), written directly.
template <typename T, int WAV, int NB, int LAY, int MODE, bool U8ONLY = false>
__device__ __forceinline__ void direct_item(const SceneArgs &s, int64_t x0, int m_s, int m_e, int b0, int lane) {
    const LaneCols c = lane_cols(x0, lane, s.W);
    DirectEmit<LAY, MODE, U8ONLY> out(s, c, b0, m_s, lane);
    walk_rows<T, WAV, NB, LAY>(s, c, x0, m_s, m_e, b0, out);
}

// Geometry of a scene's work items: strips of 128 PAN columns times runs of R MS rows.
struct ItemGrid {
    int64_t strips_x, strips_y, items;
};

__host__ __device__ inline ItemGrid item_grid(int64_t H, int64_t W, int R) {
    ItemGrid g;
    g.strips_x = (W + kWarpCols - 1) / kWarpCols;
    g.strips_y = ((H >> 1) + R - 1) / R;
    g.items = g.strips_x * g.strips_y;
    return g;
}

// Runs work item `item` of a scene on the walkers of one row layout.
template <typename T, int WAV, int NB, int LAY, int MODE, bool U8ONLY = false>
__device__ __forceinline__ void run_item(const SceneArgs &s, int64_t item, int64_t strips_x, int R, int b0, int lane) {
    const int64_t sx = item % strips_x, sy = item / strips_x;
    const int m_s = s.m_lo + (int)(sy * R);
    const int m_e = min(m_s + R, s.m_hi);
    direct_item<T, WAV, NB, LAY, MODE, U8ONLY>(s, sx * kWarpCols, m_s, m_e, b0, lane);
}

}  // namespace dwtfuse
