// Fused forward of a single scene: the grid-stride kernel.
#include "fuse_tile.cuh"
#include "launch.h"

namespace dwtfuse {

constexpr int kAltMaxBands = 6;  // widest band chunk of the shifted-row instance
// Shifted rows: neighbouring strips complete each other's sectors, and short
// items bring them there close together (rows per item 4 against the balanced
// height: 16384 x 16382 x 6 float + uint8 1948 -> 1804 us, 5000 x 5002 x 6 174
// -> 160, 3736 x 4070 x 3 49.2 -> 46.2; aligned rows gain nothing: 8192^2 x 8
// float 520 -> 526).  Not for one or two bands of floats to uint8 alone, which
// read more than they write (8190^2 D4, short -> balanced: one band 125 -> 105,
// two 150 -> 127; Haar, one 81 -> 75).
constexpr int kShiftRows = 4;

// Walker mode (paired / scalar FP32 and loads ahead, us a call) and CTA size of
// an instance.  With a float output: up to 4 bands PAN one row ahead (3736 x
// 4070 x 3 uint8 58 -> 53.5); more bands scalar columns (8192^2 x 8 uint8 to
// float + uint8 502 -> 491), floats scalar rows too (8192^2 x 8 522 -> 493, 6
// bands on shifted rows 405 -> 398), Haar, whose walker keeps no synthesised
// row, everything ahead (floats to float + uint8, 3000 x 3002 x 5 64 -> 58, 4000
// x 4002 x 6 130 -> 124; uint8 106 -> 101).  A uint8 output alone leaves the walker
// bound by instructions and load latency: paired FP32 and loads ahead as far as
// the registers go, at 8192^2: 3 bands 109 -> 103, 5 bands 155 -> 134, 7 bands
// 191 -> 175; 8 bands with 12 warps per SM whose registers hold the next row's
// inputs (208 -> 194; 7480 x 8140 193 -> 174).
template <typename T, int WAV, int NB, bool U8ONLY>
struct FwdShape {
    static constexpr int kThreads = U8ONLY && NB == 8 ? 192 : 256;
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kMode = U8ONLY    ? (NB <= 4 || NB == 8 ? kAheadPan | kAheadMs : NB <= 6 ? kAheadPan : 0)
                                 : NB <= 4 ? kAheadPan
                                 : WAV == 0 ? kAheadPan | kAheadMs
                                           : (sizeof(T) == 4 ? kScalarCol | kScalarRow : kScalarCol);
    // (8 bands: the walker without its float stores compiled to a slower
    // schedule, 193 us against 174, so that instance keeps the run-time test)
    static constexpr bool kNoFloat = U8ONLY && NB < 8;
};

// Single scene, bands [b0, b0 + NB).  Each warp takes work items
// warp, warp + total_warps, ... (grid sized to the resident capacity).
// Row layout: SHIFT kShift, else VEC kVec, else kPairs.  U8ONLY: a uint8
// output and no float one.
template <typename T, int WAV, int NB, bool U8ONLY, bool VEC, bool SHIFT>
__global__ void __launch_bounds__(FwdShape<T, WAV, NB, U8ONLY>::kThreads, 2)
fuse_fwd_kernel(const __grid_constant__ SceneArgs s, int b0, int64_t strips_x, int64_t items, int R) {
    using F = FwdShape<T, WAV, NB, U8ONLY>;
    constexpr int LAY = SHIFT ? kShift : (VEC ? kVec : kPairs);
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * F::kWarps;
    for (int64_t it = (int64_t)blockIdx.x * F::kWarps + (threadIdx.x >> 5); it < items; it += nwarps)
        run_item<T, WAV, NB, LAY, F::kMode, F::kNoFloat>(s, it, strips_x, R, b0, lane);
}

// ------------------------------------------------------------------ host side

namespace {

struct FwdFn {
    void *fn;
    int threads;
};

template <typename T, int WAV, int NB, bool U8ONLY>
FwdFn fwd_fn(int lay) {
    constexpr int kT = FwdShape<T, WAV, NB, U8ONLY>::kThreads;
    if (lay == kVec) return {reinterpret_cast<void *>(&fuse_fwd_kernel<T, WAV, NB, U8ONLY, true, false>), kT};
    if constexpr (NB <= kAltMaxBands)
        if (lay == kShift) return {reinterpret_cast<void *>(&fuse_fwd_kernel<T, WAV, NB, U8ONLY, false, true>), kT};
    if (lay == kPairs) return {reinterpret_cast<void *>(&fuse_fwd_kernel<T, WAV, NB, U8ONLY, false, false>), kT};
    return {nullptr, 0};
}

template <typename T, int WAV, bool U8ONLY>
FwdFn fwd_fn_nb(int nb, int lay) {
    switch (nb) {
        case 1: return fwd_fn<T, WAV, 1, U8ONLY>(lay);
        case 2: return fwd_fn<T, WAV, 2, U8ONLY>(lay);
        case 3: return fwd_fn<T, WAV, 3, U8ONLY>(lay);
        case 4: return fwd_fn<T, WAV, 4, U8ONLY>(lay);
        case 5: return fwd_fn<T, WAV, 5, U8ONLY>(lay);
        case 6: return fwd_fn<T, WAV, 6, U8ONLY>(lay);
        case 7: return fwd_fn<T, WAV, 7, U8ONLY>(lay);
        case 8: return fwd_fn<T, WAV, 8, U8ONLY>(lay);
        default: return {nullptr, 0};
    }
}

FwdFn fwd_kernel(const SceneArgs &s, int nb, int lay) {
    if (s.in_f32) return s.wavelet ? fwd_fn_nb<float, 1, false>(nb, lay) : fwd_fn_nb<float, 0, false>(nb, lay);
    if (s.out_f32 == nullptr)
        return s.wavelet ? fwd_fn_nb<uint8_t, 1, true>(nb, lay) : fwd_fn_nb<uint8_t, 0, true>(nb, lay);
    return s.wavelet ? fwd_fn_nb<uint8_t, 1, false>(nb, lay) : fwd_fn_nb<uint8_t, 0, false>(nb, lay);
}

}  // namespace

cudaError_t launch_fuse(const SceneArgs &s, int R, int blocks_per_sm, cudaStream_t stream) {
    // Scenes with a float output where it pays: the staged kernel (its float
    // rows go out as bulk copies).
    if (fuse_staging() && fuse_staged_applies(s)) return launch_fuse_staged(s, R, stream);
    // Bands go in chunks of up to 8; the shifted-row instance (W % 4 == 2)
    // holds more live registers per band and takes balanced chunks of <= 6;
    // a band-chunk knob (autotuner) caps both, in balanced chunks.
    const bool alt = s.alt != 0 && s.a4 == 0;
    const int knob = fwd_band_chunk();
    int cap = alt ? kAltMaxBands : kChunkBands;
    if (knob > 0 && knob < cap) cap = knob;
    const int nchunks = (s.bands + cap - 1) / cap;
    const int chunk = (alt || knob > 0) ? (s.bands + nchunks - 1) / nchunks : kChunkBands;
    for (int b0 = 0; b0 < s.bands; b0 += chunk) {
        const int nb = s.bands - b0 < chunk ? s.bands - b0 : chunk;
        const FwdFn k = fwd_kernel(s, nb, row_layout(s.a4, s.alt));
        void *fn = k.fn;
        const int warps = k.threads / 32;
        if (fn == nullptr) return cudaErrorInvalidValue;
        int occ = 0;
        cudaError_t e = resident_blocks(fn, k.threads, &occ);
        if (e != cudaSuccess) return e;
        if (blocks_per_sm > 0 && blocks_per_sm < occ) occ = blocks_per_sm;
        int sms = 0;
        e = sm_count(&sms);
        if (e != cudaSuccess) return e;
        const int64_t cap = (int64_t)sms * occ;
        // Items cover the MS rows [m_lo, m_hi) (all of them for a whole scene).
        const int64_t rows2 = 2 * (int64_t)(s.m_hi - s.m_lo);
        int Rl = R;
        if (Rl <= 0) {
            Rl = balanced_rows((s.W + kWarpCols - 1) / kWarpCols, rows2 / 2, cap * warps);
            // (the least output bytes a pixel for which they pay, against the PAN bytes that
            // short items read again)
            const int px_out = nb * ((s.out_f32 ? 4 : 0) + (s.out_u8 ? 1 : 0)), px_pan = s.in_f32 ? 4 : 1;
            if (alt && 2 * px_out > px_pan && Rl > kShiftRows) Rl = kShiftRows;
        }
        const ItemGrid g = item_grid(rows2, s.W, Rl);
        const int64_t need = (g.items + warps - 1) / warps;
        const unsigned grid = (unsigned)(need < cap ? need : cap);
        if (grid == 0) continue;
        SceneArgs sa = s;
        int64_t strips_x = g.strips_x, items = g.items;
        void *args[] = {&sa, (void *)&b0, &strips_x, &items, &Rl};
        e = cudaLaunchKernel(fn, dim3(grid), dim3(k.threads), args, 0, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dwtfuse
