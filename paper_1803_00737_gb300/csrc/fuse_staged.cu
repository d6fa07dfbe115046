// Fused forward with the float output rows written by the bulk copy engine.
//
// The arithmetic is that of fuse_fwd.cu (Sec. 2, Eq. 1-16, through the warp
// walkers of fuse_tile.cuh); what changes is how the float rows reach HBM.
// A CTA of 8 warps owns a strip of 1024 PAN columns (its warps' 128-column
// strips side by side) and walks down its MS rows in step: for every MS row
// the lanes put their 4 float pixels of both PAN rows of every band into a
// shared-memory slot, the CTA meets at one barrier, and 2 NB threads each
// issue one cp.async.bulk (shared::cta -> global) of a 4 KB row segment.  The
// CTA's rows alternate between two slots (a count carried across work items,
// so consecutive rows never share one); the issuing threads wait
// (cp.async.bulk.wait_group.read) for their previous copies before the
// barrier of the next row, when those reads are long done, so the slot a row
// overwrites is free.  uint8 outputs keep the per-lane stores.
//
// Why: a warp's 16-byte-per-lane stores send a row segment to L2 as 4 line
// requests (5 when the row starts off the 128-byte line grid, with the
// segment's end sectors shared between two warps' requests); the bulk copy
// moves 4 KB per request stream and leaves only the CTA strip ends partial.
// Measured (16384 rows, 6 bands, float32 + uint8, CUDA events): W = 16384
// 6168 -> 6538 GB/s, W = 16380 5117 -> 6261, W = 16376 5729 -> 6307,
// W = 4092 5364 -> 6137.  A single slot with a second barrier per row (wait
// for the copies' reads, then release the slot) ran 5180-5330 GB/s on every
// width.
//
// Used for single scenes (fuse_staged_applies) in chunks of at most
// kStagedMaxBands bands (two slots of 6 bands x 2 rows x 4 KB = 96 KB, two
// CTAs per SM; the band-chunk knob splits them further).  A bulk copy starts
// on a 16-byte boundary and moves a multiple of 16 bytes: rows on the 16-byte
// grid go out whole; on shifted rows (W % 4 == 2) the slot's odd rows lie 2
// floats in, and the pairs at a row segment's ends go out as plain stores.
#include "fuse_tile.cuh"
#include "launch.h"

namespace dwtfuse {

namespace {

constexpr int kStThreads = 256;
constexpr int kStWarps = kStThreads / 32;
constexpr int kStCols = kStWarps * kWarpCols;  // 1024 PAN columns per CTA strip

__device__ __forceinline__ unsigned st_smem(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bulk_out(float *dst, const float *src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(st_smem(src)), "r"(bytes)
                 : "memory");
}
// The issuing threads' bulk copies have read their shared-memory source.
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
}

// The CTA's row barrier.  An emitter's row_end is instantiated in the inner-strip
// and the edge-strip walker, and the warps of one CTA run both: every thread
// (idle lanes too) arrives once per MS row, at one of several barrier
// instructions.  PTX counts the arrivals per barrier number, whichever
// instruction they come from, and without .aligned asks nothing of a warp's
// convergence; __syncthreads() is defined only where the whole block takes the
// same side of every condition around it.
__device__ __forceinline__ void row_barrier() { asm volatile("barrier.sync 0;\n" ::: "memory"); }

// Floats between the slot's rows: with SHIFT a row's pixels start 0 (even rows)
// or 2 (odd rows) floats in, like the image row past its 16-byte boundary.
template <bool SHIFT>
constexpr int kStRow = kStCols + (SHIFT ? 8 : 0);

template <int WAV, int NB, bool SHIFT, bool LATE>
struct StagedEmit {
    static constexpr int kRow = kStRow<SHIFT>, kLay = SHIFT ? kShift : kVec;
    // Up to 4 bands: the next row's inputs loaded ahead (8192^2 x 3 208 -> 184
    // us).  More: nothing ahead, D4 with scalar synthesis (its registers), Haar
    // paired (loads ahead: 8190^2 x 6 uint8 to float 282 -> 306).
    static constexpr int kMode = NB <= 4 ? kAheadPan | kAheadMs : WAV ? kScalarCol | kScalarRow : 0;
    const SceneArgs &s;
    const LaneCols &c;
    float *buf;    // two slots of [NB][2][kRow] floats
    int64_t X0;    // first column of the CTA strip
    int ncols;     // columns of the strip inside the image (even; a multiple of 4 but for SHIFT)
    int lane;
    int b0;        // first band of the launch's chunk
    int *rowc;     // the CTA's row count: row k fills slot k & 1
    bool hu;       // uint8 output wanted
    uint8_t *u;    // its band b0, the current MS row's first image row, column x
    uint32_t w8[LATE ? NB : 1][2];  // LATE: the row's uint8 words

    __device__ __forceinline__ float *slot() const { return buf + (*rowc & 1) * (NB * 2 * kRow); }

    template <typename M>
    __device__ __forceinline__ void band(int b, const float *v0, const float *v1, M, M) {
        if (LATE) {
            if (hu) {
                w8[LATE ? b : 0][0] = pack4u8(v0);
                w8[LATE ? b : 0][1] = pack4u8(v1);
            }
        } else {
            u += b ? s.out_plane : 0;
        }
        if (c.active) {
            float *row = slot() + b * 2 * kRow + (c.x - (int)X0);
            *reinterpret_cast<float4 *>(row) = make_float4(v0[0], v0[1], v0[2], v0[3]);
            if (SHIFT) {
                *reinterpret_cast<float2 *>(row + kRow + 2) = make_float2(v1[0], v1[1]);
                *reinterpret_cast<float2 *>(row + kRow + 4) = make_float2(v1[2], v1[3]);
            } else {
                *reinterpret_cast<float4 *>(row + kRow) = make_float4(v1[0], v1[1], v1[2], v1[3]);
            }
        }
        if (!LATE && hu) store_rows(u, pack4u8(v0), pack4u8(v1));
    }

    __device__ __forceinline__ void store_rows(uint8_t *q, uint32_t w0, uint32_t w1) const {
        store_u8<kLay>(q, c, lane, false, w0);
        store_u8<kLay>(q + s.W, c, lane, true, w1);
    }

    template <int>
    __device__ __forceinline__ void row_end(int m, uint32_t, uint32_t) {
        // Make this thread's shared-memory writes visible to the bulk copy engine.
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        const int t = threadIdx.x;
        if (t < 2 * NB) bulk_wait_read();  // row m-1's copies: the slot row m+1 will fill
        row_barrier();
        if (t < 2 * NB) {
            const int b = t >> 1, r = t & 1;
            const int64_t y = 2 * (int64_t)(m - s.m_lo) + r;
            float *dst = s.out_f32 + (int64_t)(b0 + b) * s.out_plane + y * s.W + X0;
            const float *src = slot() + (b * 2 + r) * kRow;
            if (SHIFT) {
                // The pixel pairs before the first and after the last 16-byte
                // boundary by plain stores, what lies between as one copy.
                int n = ncols;
                if (r) {
                    *reinterpret_cast<float2 *>(dst) = *reinterpret_cast<const float2 *>(src + 2);
                    dst += 2;
                    src += 4;
                    n -= 2;
                }
                if (n & 2)
                    *reinterpret_cast<float2 *>(dst + (n & ~3)) = *reinterpret_cast<const float2 *>(src + (n & ~3));
                if (n >= 4) bulk_out(dst, src, (unsigned)(n & ~3) * 4u);
            } else {
                bulk_out(dst, src, (unsigned)ncols * 4u);
            }
            asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
        }
        if (LATE) {
            if (hu) {
                uint8_t *q = u;
#pragma unroll
                for (int b = 0; b < (LATE ? NB : 1); ++b) {
                    store_rows(q, w8[b][0], w8[b][1]);
                    q += s.out_plane;
                }
            }
            u += 2 * s.W;
        } else {
            u += 2 * s.W - (NB - 1) * s.out_plane;
        }
        ++*rowc;
    }
};

// One CTA item: columns [X0, X0 + 1024), MS rows [m_s, m_e), bands
// [b0, b0 + NB).  Every thread of the CTA calls it, with the same row count.
template <typename T, int WAV, int NB, bool SHIFT, bool LATE>
__device__ __forceinline__ void staged_item(const SceneArgs &s, float *buf, int64_t X0, int m_s, int m_e, int b0,
                                            int *rowc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t x0 = X0 + (int64_t)warp * kWarpCols;
    const LaneCols c = lane_cols(x0, lane, s.W);  // warps past W: idle lanes
    const int ncols = (int)min((int64_t)kStCols, s.W - X0);
    uint8_t *u = s.out_u8 + (int64_t)b0 * s.out_plane + (int64_t)(2 * (m_s - s.m_lo)) * s.W + c.x;
    StagedEmit<WAV, NB, SHIFT, LATE> out{s, c, buf, X0, ncols, lane, b0, rowc, s.out_u8 != nullptr, u};
    walk_rows<T, WAV, NB, SHIFT ? kShift : kVec>(s, c, x0, m_s, m_e, b0, out);
}

__device__ __forceinline__ void bulk_drain() {
    if (threadIdx.x < 2 * kStagedMaxBands) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
}

}  // namespace

// Single scene, bands [b0, b0 + NB); CTA items it = blockIdx.x, + gridDim.x, ...
template <typename T, int WAV, int NB, bool SHIFT, bool LATE>
__global__ void __launch_bounds__(kStThreads, 2)
fuse_staged_kernel(const __grid_constant__ SceneArgs s, int b0, int64_t strips_cta, int64_t items, int R) {
    extern __shared__ __align__(128) float st_buf[];
    int rowc = 0;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int64_t sx = it % strips_cta, sy = it / strips_cta;
        const int m_s = s.m_lo + (int)(sy * R);
        staged_item<T, WAV, NB, SHIFT, LATE>(s, st_buf, sx * kStCols, m_s, min(m_s + R, s.m_hi), b0, &rowc);
    }
    bulk_drain();
}

namespace {

template <typename T, int WAV, int NB>
void *st_fn_nb(bool shift, bool late) {
    if constexpr (NB == 6 && (WAV || sizeof(T) == 1))
        if (late) return reinterpret_cast<void *>(&fuse_staged_kernel<T, WAV, NB, false, true>);
    return shift ? reinterpret_cast<void *>(&fuse_staged_kernel<T, WAV, NB, true, false>)
                 : reinterpret_cast<void *>(&fuse_staged_kernel<T, WAV, NB, false, false>);
}

template <typename T, int WAV>
void *st_fn(int nb, bool shift, bool late) {
    switch (nb) {
        case 1: return st_fn_nb<T, WAV, 1>(shift, late);
        case 2: return st_fn_nb<T, WAV, 2>(shift, late);
        case 3: return st_fn_nb<T, WAV, 3>(shift, late);
        case 4: return st_fn_nb<T, WAV, 4>(shift, late);
        case 5: return st_fn_nb<T, WAV, 5>(shift, late);
        case 6: return st_fn_nb<T, WAV, 6>(shift, late);
        default: return nullptr;
    }
}

constexpr int staged_smem(int nb, bool shift) {
    return 2 * nb * 2 * (shift ? kStRow<true> : kStRow<false>) * (int)sizeof(float);
}

}  // namespace

// The staged kernel pays where a CTA's 8 warps, which meet at a barrier every
// MS row, rarely wait for one another: nearly whole 1024-column strips (idle
// warps in a ragged last strip are lost time).  Up to 6 bands on aligned rows:
// at every size (16384 x 4092 x 6 5364 -> 6137 GB/s against the warp kernel).
// Shifted rows, and uint8 scenes of more bands (balanced chunks of at most 6,
// PAN read once per chunk): where the output is many times the L2
// (kStagedLarge bytes); smaller ones run faster item by item.  us, warp ->
// staged: 16384 x 16382 x 6 1789 -> 1542, 8190^2 x 8 560 -> 500, 8190^2 x 3 230
// -> 197, 8192 x 8140 x 8 554 -> 504, 16384^2 x 8 1952 -> 1910, 8192^2 x 12 733
// -> 675; below the line 3736 x 4070 x 3 47 -> 51, 3000 x 2998 x 5 48 -> 55,
// 4096^2 x 8 float 102 -> 107.  Float scenes of more than 6 aligned bands read
// four times the PAN bytes per chunk and stay on the warp kernel; so do, for
// float alone, the 7 and 8 aligned bands that D4 takes in one warp launch, 8 up to
// four times that line (staged -> warp: 8192^2 x 7 349 -> 335, 16384^2 x 7 1362 ->
// 1333, 4096 x 8192 x 8 197 -> 194, 8192^2 x 8 381 -> 378; 12000 x 12288 x 8 827 ->
// 830, 16384^2 x 8 1491 -> 1515; Haar 8192^2 x 7 339 -> 350).  The same CTA
// items in the batched launch ran slower than its warp items on every scene
// class tried (46 scenes on the grid: 5356 -> 4651 GB/s; with the next item
// fetched during the current one and 64-row items: 4644), so the batched
// launch keeps warp items.
constexpr int64_t kStagedLarge = 700000000;

bool fuse_staged_applies(const SceneArgs &s) {
    if ((s.a4 == 0 && s.alt == 0) || s.out_f32 == nullptr) return false;
    const bool more = s.bands > kStagedMaxBands;
    if (s.a4 == 0 || more) {
        if (s.a4 != 0 && s.in_f32) return false;
        const int64_t px = 2 * (int64_t)(s.m_hi - s.m_lo) * s.W * s.bands, bytes = px * (s.out_u8 ? 5 : 4);
        if (bytes < kStagedLarge) return false;
        if (s.a4 != 0 && s.wavelet && s.out_u8 == nullptr &&
            (s.bands < kChunkBands || (s.bands == kChunkBands && bytes < 4 * kStagedLarge)))
            return false;
    }
    const int64_t strips = (s.W + kStCols - 1) / kStCols;
    return (strips * kStCols - s.W) * 8 <= strips * kStCols;
}

// Whether the uint8 pixels are stored after the float rows' copies are issued,
// behind the row barrier, instead of band by band before it.  Only 6 bands on
// aligned rows gain by it, and not all of them.  us, before -> behind, float +
// uint8: D4 on the 128-byte line grid 16384^2 1378 -> 1334, 8192^2 347 -> 337;
// off that grid uint8 3000 x 4092 69.7 -> 70.5, float 82.8 -> 85.5, 4958 x 7932
// 258 -> 263; Haar uint8 8192^2 365 -> 353, 4958 x 7932 229 -> 214; Haar float
// 4958 x 7932 262 -> 280.  Five bands lose (D4 4096^2 76.2 -> 80.0, 12000 x 12284
// 645 -> 687), and so do shifted rows (8190^2 x 6 356 -> 389).
static bool staged_late(const SceneArgs &s, int nb) {
    return nb == 6 && s.a4 != 0 && s.out_u8 != nullptr && (s.wavelet ? s.W % 32 == 0 : s.in_f32 == 0);
}

static int64_t staged_strips(int64_t W) { return (W + kStCols - 1) / kStCols; }

cudaError_t launch_fuse_staged(const SceneArgs &s, int R, cudaStream_t stream) {
    int cap = kStagedMaxBands;
    const int knob = fwd_band_chunk();
    if (knob > 0 && knob < cap) cap = knob;
    const int nchunks = (s.bands + cap - 1) / cap;
    const int chunk = (s.bands + nchunks - 1) / nchunks;  // balanced
    int sms = 0;
    cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    for (int b0 = 0; b0 < s.bands; b0 += chunk) {
        const int nb = s.bands - b0 < chunk ? s.bands - b0 : chunk;
        const bool shift = s.a4 == 0;
        const bool late = staged_late(s, nb);
        void *fn = s.in_f32 ? (s.wavelet ? st_fn<float, 1>(nb, shift, late) : st_fn<float, 0>(nb, shift, late))
                            : (s.wavelet ? st_fn<uint8_t, 1>(nb, shift, late) : st_fn<uint8_t, 0>(nb, shift, late));
        if (fn == nullptr) return cudaErrorInvalidValue;
        const int smem = staged_smem(nb, shift);
        int occ = 0;
        e = resident_blocks_smem(fn, kStThreads, smem, &occ);
        if (e != cudaSuccess) return e;
        const int64_t capc = (int64_t)sms * occ;
        const int64_t rows = (int64_t)(s.m_hi - s.m_lo);
        const int64_t strips = staged_strips(s.W);
        int Rl = R;
        if (Rl <= 0) Rl = balanced_rows(strips, rows, capc, 128);
        const int64_t items = strips * ((rows + Rl - 1) / Rl);
        const unsigned grid = (unsigned)(items < capc ? items : capc);
        if (grid == 0) continue;
        SceneArgs sa = s;
        int b0v = b0;
        int64_t sv = strips, iv = items;
        void *args[] = {&sa, &b0v, &sv, &iv, &Rl};
        e = cudaLaunchKernel(fn, dim3(grid), dim3(kStThreads), args, (size_t)smem, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace dwtfuse
