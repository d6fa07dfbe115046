// Fused forward of a single scene: the grid-stride kernel.
#include "fuse_tile.cuh"
#include "launch.h"

namespace dwtfuse {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kAltMaxBands = 6;  // widest band chunk of the shifted-row instance
// Shifted rows: neighbouring strips complete each other's sectors, and short
// items bring them there close together (rows per item 4 against the balanced
// height: 16384 x 16382 x 6 float + uint8 1948 -> 1804 us, 5000 x 5002 x 6 174
// -> 160, 3736 x 4070 x 3 49.2 -> 46.2; aligned rows gain nothing: 8192^2 x 8
// float 520 -> 526).
constexpr int kShiftRows = 4;

// Walker mode (paired / scalar FP32 and loads ahead, us a call): up to 4 bands
// PAN one row ahead (3736 x 4070 x 3 uint8 58 -> 53.5); more bands scalar
// columns (8192^2 x 8 uint8 to float + uint8 502 -> 491, to uint8 alone 205 ->
// 211), floats scalar rows too (8192^2 x 8 522 -> 493, 6 bands on shifted rows
// 405 -> 398).
template <typename T, int NB>
constexpr int kFwdMode = NB <= 4 ? kAheadPan : (sizeof(T) == 4 ? kScalarCol | kScalarRow : kScalarCol);

// Single scene, bands [b0, b0 + NB).  Each warp takes work items
// warp, warp + total_warps, ... (grid sized to the resident capacity).
// Row layout: SHIFT kShift, else VEC kVec, else kPairs.
template <typename T, int WAV, int NB, bool VEC, bool SHIFT>
__global__ void __launch_bounds__(kThreads, 2)
fuse_fwd_kernel(const __grid_constant__ SceneArgs s, int b0, int64_t strips_x, int64_t items, int R) {
    constexpr int LAY = SHIFT ? kShift : (VEC ? kVec : kPairs);
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * kWarps;
    for (int64_t it = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); it < items; it += nwarps)
        run_item<T, WAV, NB, LAY, kFwdMode<T, NB>>(s, it, strips_x, R, b0, lane);
}

// ------------------------------------------------------------------ host side

namespace {

template <typename T, int WAV, int NB>
void *fwd_fn(int lay) {
    if (lay == kVec) return reinterpret_cast<void *>(&fuse_fwd_kernel<T, WAV, NB, true, false>);
    if constexpr (NB <= kAltMaxBands)
        if (lay == kShift) return reinterpret_cast<void *>(&fuse_fwd_kernel<T, WAV, NB, false, true>);
    return lay == kPairs ? reinterpret_cast<void *>(&fuse_fwd_kernel<T, WAV, NB, false, false>) : nullptr;
}

template <typename T, int WAV>
void *fwd_fn_nb(int nb, int lay) {
    switch (nb) {
        case 1: return fwd_fn<T, WAV, 1>(lay);
        case 2: return fwd_fn<T, WAV, 2>(lay);
        case 3: return fwd_fn<T, WAV, 3>(lay);
        case 4: return fwd_fn<T, WAV, 4>(lay);
        case 5: return fwd_fn<T, WAV, 5>(lay);
        case 6: return fwd_fn<T, WAV, 6>(lay);
        case 7: return fwd_fn<T, WAV, 7>(lay);
        case 8: return fwd_fn<T, WAV, 8>(lay);
        default: return nullptr;
    }
}

void *fwd_kernel_ptr(bool f32, int wav, int nb, int lay) {
    if (f32) return wav ? fwd_fn_nb<float, 1>(nb, lay) : fwd_fn_nb<float, 0>(nb, lay);
    return wav ? fwd_fn_nb<uint8_t, 1>(nb, lay) : fwd_fn_nb<uint8_t, 0>(nb, lay);
}

}  // namespace

cudaError_t launch_fuse(const SceneArgs &s, int R, int blocks_per_sm, cudaStream_t stream) {
    // Large scenes whose rows lie on the 16-byte grid with a float output: the
    // staged kernel (its float rows go out as bulk copies).
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
        void *fn = fwd_kernel_ptr(s.in_f32 != 0, s.wavelet, nb, row_layout(s.a4, s.alt));
        if (fn == nullptr) return cudaErrorInvalidValue;
        int occ = 0;
        cudaError_t e = resident_blocks(fn, kThreads, &occ);
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
            Rl = balanced_rows((s.W + kWarpCols - 1) / kWarpCols, rows2 / 2, cap * kWarps);
            if (alt && Rl > kShiftRows) Rl = kShiftRows;
        }
        const ItemGrid g = item_grid(rows2, s.W, Rl);
        const int64_t need = (g.items + kWarps - 1) / kWarps;
        const unsigned grid = (unsigned)(need < cap ? need : cap);
        if (grid == 0) continue;
        SceneArgs sa = s;
        int64_t strips_x = g.strips_x, items = g.items;
        void *args[] = {&sa, (void *)&b0, &strips_x, &items, &Rl};
        e = cudaLaunchKernel(fn, dim3(grid), dim3(kThreads), args, 0, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dwtfuse
