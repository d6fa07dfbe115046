// Batched fused forward: the persistent kernel fed by a device-side work queue.
#include <algorithm>

#include "fuse_tile.cuh"
#include "launch.h"

namespace dwtfuse {

constexpr int kBatchNarrowBands = 4;  // instance for entries of at most 4 bands
constexpr int kBatchLightBands = 3;   // float instance for entries of light bodies alone
// A float body whose registers leave room for 20 warps per SM.
__host__ __device__ constexpr bool light_body(int wavelet, int bands) {
    return bands == 1 || (wavelet == 0 && bands <= kBatchLightBands);
}
constexpr int kSceneBytes = (int)((sizeof(SceneArgs) + 15) / 16 * 16);

// Threads per CTA (two CTAs per SM), walker mode and shared memory (per warp, a
// copy of its item's scene) of an instance.  Entries of at most 4 bands:
// uint8 20 warps per SM at up to 96 registers (24 uneven scenes of 3-8 bands,
// 256..4096 px: 719 us a call against 730 with 16 warps at 128), float 16
// warps with the next row's inputs loaded ahead (forward + backward of
// 8 x 4096^2 x 4: 1086 us a pass against 1129 with 20 warps, where that
// spills, and 1101 with 16 and no loads ahead), or 20 warps where all entries are
// Haar of at most 3 bands or have one band (4 x 4096^2, 16 -> 20 warps: Haar x 1 125
// -> 116, x 2 170 -> 159, x 3 213 -> 202, D4 x 1 134 -> 122; D4 x 2 and x 3 spill
// there, 181 -> 202, 237 -> 284).  More bands, 16 warps: floats
// with scalar synthesis (4 x 4096^2 x 8 570 -> 480 us a call, 8 x 2048^2 x 8
// 298 -> 248; paired, the walker spills more), uint8 paired with PAN ahead (24
// uneven scenes to uint8 469 -> 464) but for 8 bands of D4, which then spill 212
// bytes a thread (to float 4 x 4096^2 430 -> 377, 16 x 1000 x 1004 120 -> 108).
template <typename T, int MAXB>
struct BatchShape {
    static constexpr bool kNarrow = MAXB <= kBatchNarrowBands, kFloat = sizeof(T) == 4;
    static constexpr bool kLight = kFloat && MAXB == kBatchLightBands;
    static constexpr int kThreads = kNarrow && (!kFloat || kLight) ? 320 : 256;
    template <int WAV, int NB>
    static constexpr int kMode = kNarrow  ? (kFloat ? kAheadPan | kAheadMs : 0)
                                 : kFloat ? kScalarCol | kScalarRow
                                          : (WAV && NB == 8 ? kScalarCol : kAheadPan);
    static constexpr int kSmem = kThreads / 32 * kSceneBytes;
    static constexpr int kMinBands = kNarrow ? 1 : kBatchNarrowBands + 1;  // fewer: the narrow instance's entries
};

extern __shared__ __align__(16) unsigned char batch_smem[];

// One item of a scene with NB bands: the scene is the warp's shared-memory
// copy (in the kernel's parameter block it would be read at run-time offsets
// and its members held in registers).  A function of its own, not inlined:
// each of an instance's bodies gets its own register allocation (all inlined
// in one kernel they spilled up to 0.5 KB a thread).  D4 bodies still report
// spills, in bytes of stores a thread: uint8 12-44 up to 4 bands, 36-104 with 5-8,
// float up to 12 and up to 52 (the kernels themselves 4-12; Haar none).  Not
// measured: how many of them are registers saved for the caller, once an item.
template <typename T, int WAV, int NB, int LAY, int MODE>
static __device__ __noinline__ void batch_body(int x0, int m_s, int m_e) {
    const SceneArgs &s = *reinterpret_cast<const SceneArgs *>(batch_smem + (threadIdx.x >> 5) * kSceneBytes);
    direct_item<T, WAV, NB, LAY, MODE>(s, x0, m_s, m_e, 0, threadIdx.x & 31);
}

// The item by its entry's row layout (entries on shifted rows hold at most
// kBatchAltMaxBands bands: the table splits them or clears alt).
template <typename T, int WAV, int NB, int MODE>
static __device__ __forceinline__ void batch_item(const SceneArgs &s, int x0, int m_s, int m_e) {
    if (s.a4) {
        batch_body<T, WAV, NB, kVec, MODE>(x0, m_s, m_e);
        return;
    }
    if constexpr (NB <= kBatchAltMaxBands) {
        if (s.alt) {
            batch_body<T, WAV, NB, kShift, MODE>(x0, m_s, m_e);
            return;
        }
    }
    batch_body<T, WAV, NB, kPairs, MODE>(x0, m_s, m_e);
}

// Batched: every warp pulls the next item index from `queue[0]`; item ranges
// of the scenes are given by the prefix sums item_start[].  A warp whose
// scene table entry fails its checks records DWTFUSE_EDEVICE in status[0].
// An instance serves one input type and at most MAXB bands per entry.
template <typename T, int MAXB>
__global__ void __launch_bounds__(BatchShape<T, MAXB>::kThreads, 2)
fuse_batched_kernel(const __grid_constant__ BatchTable t, unsigned long long *queue, int *status) {
    uint32_t *copy = reinterpret_cast<uint32_t *>(batch_smem + (threadIdx.x >> 5) * kSceneBytes);
    const int lane = threadIdx.x & 31;
    const unsigned long long total = (unsigned long long)t.item_start[t.n];
    int have = -1;  // scene the warp's copy holds
    for (;;) {
        unsigned long long it = 0;
        if (lane == 0) it = atomicAdd(queue, 1ull);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= total) break;
        int lo = 0, hi = t.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((unsigned long long)t.item_start[mid] <= it) lo = mid; else hi = mid - 1;
        }
        const SceneArgs &s = t.scenes[lo];
        using Shape = BatchShape<T, MAXB>;
        if (s.bands < Shape::kMinBands || s.bands > MAXB || (s.in_f32 != 0) != (sizeof(T) == 4) ||
            (Shape::kLight && !light_body(s.wavelet, s.bands))) {
            if (lane == 0) atomicCAS(status, 0, 7);
            continue;
        }
        if (have != lo) {
            __syncwarp();  // every lane is done with the previous scene
            const uint32_t *src = reinterpret_cast<const uint32_t *>(&s);
            for (int k = lane; k < (int)(sizeof(SceneArgs) / 4); k += 32) copy[k] = src[k];
            have = lo;
            __syncwarp();
        }
        const int64_t local = (int64_t)(it - (unsigned long long)t.item_start[lo]);
        const int64_t sx = local % t.strips_x[lo], sy = local / t.strips_x[lo];
        const int x0 = (int)(sx * kWarpCols), m_s = s.m_lo + (int)(sy * t.R), m_e = min(m_s + t.R, s.m_hi);
#define DWTFUSE_CASE(NBV)                                                                        \
    case NBV:                                                                                    \
        if constexpr (NBV >= Shape::kMinBands && NBV <= MAXB) {                                  \
            if (!s.wavelet) {                                                                    \
                batch_item<T, 0, NBV, Shape::template kMode<0, NBV>>(s, x0, m_s, m_e);           \
            } else if constexpr (!Shape::kLight || light_body(1, NBV)) {                         \
                batch_item<T, 1, NBV, Shape::template kMode<1, NBV>>(s, x0, m_s, m_e);           \
            }                                                                                    \
        }                                                                                        \
        break;
        switch (s.bands) {
            DWTFUSE_CASE(1) DWTFUSE_CASE(2) DWTFUSE_CASE(3) DWTFUSE_CASE(4)
            DWTFUSE_CASE(5) DWTFUSE_CASE(6) DWTFUSE_CASE(7) DWTFUSE_CASE(8)
            default: break;
        }
#undef DWTFUSE_CASE
    }
}

namespace {

// Launches one instance over table t (entries of one input type and width
// class).  clear: bytes of the queue word(s) to zero first (the queue counter
// and status word, or only the counter so that a status an earlier launch of
// the same call recorded survives).
struct BatchFn {
    void *fn;
    int threads, smem;
};
template <typename T, int MAXB>
BatchFn batch_fn() {
    return {reinterpret_cast<void *>(&fuse_batched_kernel<T, MAXB>), BatchShape<T, MAXB>::kThreads,
            BatchShape<T, MAXB>::kSmem};
}

cudaError_t launch_table(const BatchTable &t, unsigned long long *queue, int *status, int blocks_per_sm,
                         size_t clear, cudaStream_t stream) {
    const bool f32 = t.scenes[0].in_f32 != 0, narrow = t.scenes[0].bands <= kBatchNarrowBands;
    bool light = f32;
    for (int i = 0; light && i < t.n; ++i) light = light_body(t.scenes[i].wavelet, t.scenes[i].bands);
    const BatchFn k = light    ? batch_fn<float, kBatchLightBands>()
                      : narrow ? (f32 ? batch_fn<float, kBatchNarrowBands>() : batch_fn<uint8_t, kBatchNarrowBands>())
                               : (f32 ? batch_fn<float, kBatchMaxBands>() : batch_fn<uint8_t, kBatchMaxBands>());
    void *fn = k.fn;
    const int threads = k.threads, smem = k.smem;
    int occ = 0;
    cudaError_t e = resident_blocks_smem(fn, threads, smem, &occ);
    if (e != cudaSuccess) return e;
    if (blocks_per_sm > 0 && blocks_per_sm < occ) occ = blocks_per_sm;
    int sms = 0;
    e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(queue, 0, clear, stream);
    if (e != cudaSuccess) return e;
    const int64_t total = t.item_start[t.n];
    const int64_t need = (total + threads / 32 - 1) / (threads / 32);
    const int64_t cap = (int64_t)sms * occ;
    const unsigned grid = (unsigned)(need < cap ? need : cap);
    if (grid == 0) return cudaSuccess;
    void *args[] = {const_cast<BatchTable *>(&t), &queue, &status};
    return cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, (size_t)smem, stream);
}

// MS rows per item of a launch over table t: a tenth of a warp's
// share of the rows (16 warps per SM), at most kDefaultRows, so that the
// queue's last items leave little of the GPU idle (24 uneven scenes, 94 and 75
// rows a warp in the two launches: 32 rows 721 us a call, 16 rows 653, 8 rows
// 644), and down to single rows, so that small tables still reach every warp
// (8 scenes of 256..600 px: 106 -> 40 us); large uniform tables keep tall
// items (8 x 4096^2 x 4 float, 215 rows a warp: 24 rows 521 us, 8 rows 533).
int default_rows(const BatchTable &t, int sms) {
    double rows = 0;
    for (int i = 0; i < t.n; ++i) rows += (double)t.strips_x[i] * (t.scenes[i].m_hi - t.scenes[i].m_lo);
    const double share = rows / (16.0 * sms), low = share < 4 ? share : 4;
    const double r = share / 10 > low ? share / 10 : low;
    return r < 1 ? 1 : (r > kDefaultRows ? kDefaultRows : (int)(r + 0.5));
}

// Bands, wavelet and row layout of an entry: the item body it runs.
int body_of(const SceneArgs &s) { return (s.bands * 2 + s.wavelet) * 3 + row_layout(s.a4, s.alt); }

// The entries of t of input type f32 and width class narrow (at most
// kBatchNarrowBands bands or more), those of one body together: warps of an SM
// work on neighbouring items, so they run one or two bodies at a time and share
// their instructions (24 uneven scenes in the caller's order: 768 us,
// instruction fetch 1.9 of 12 stall cycles per issue; sorted 719 us).
void split_table(const BatchTable &t, bool f32, bool narrow, BatchTable *o) {
    int order[kMaxScenes], m = 0;
    for (int i = 0; i < t.n; ++i)
        if ((t.scenes[i].in_f32 != 0) == f32 && (t.scenes[i].bands <= kBatchNarrowBands) == narrow) order[m++] = i;
    std::stable_sort(order, order + m, [&](int a, int b) { return body_of(t.scenes[a]) > body_of(t.scenes[b]); });
    o->n = m;
    o->R = t.R;
    for (int j = 0; j < m; ++j) {
        o->scenes[j] = t.scenes[order[j]];
        o->strips_x[j] = t.strips_x[order[j]];
    }
}

// Item height (where the caller left it open) and item ranges of a launch's table.
void lay_out_items(BatchTable *t, int sms) {
    if (t->R <= 0) t->R = default_rows(*t, sms);
    t->item_start[0] = 0;
    for (int j = 0; j < t->n; ++j) {
        const SceneArgs &s = t->scenes[j];
        t->item_start[j + 1] = t->item_start[j] + t->strips_x[j] * ((s.m_hi - s.m_lo + t->R - 1) / t->R);
    }
}

}  // namespace

// One launch per input type and width class in the table, the wide ones first.
// A table of one body (a batch tensor) is launched as it is: copying its
// entries cost 4 us of a call (128 scenes of 128^2 x 3: 41 -> 45 us).
cudaError_t launch_fuse_batched(BatchTable &t, unsigned long long *queue, int *status,
                                int blocks_per_sm, cudaStream_t stream) {
    int count[2][2] = {};
    bool one_body = true;
    for (int i = 0; i < t.n; ++i) {
        ++count[t.scenes[i].in_f32 != 0][t.scenes[i].bands <= kBatchNarrowBands];
        one_body = one_body && t.scenes[i].in_f32 == t.scenes[0].in_f32 && body_of(t.scenes[i]) == body_of(t.scenes[0]);
    }
    int sms = 0;
    const cudaError_t es = sm_count(&sms);
    if (es != cudaSuccess) return es;
    if (one_body && t.n > 0) {
        lay_out_items(&t, sms);
        return launch_table(t, queue, status, blocks_per_sm, kQueueBytes, stream);
    }
    static thread_local BatchTable part;
    size_t clear = kQueueBytes;
    for (int kind = 0; kind < 4; ++kind) {
        const bool narrow = kind >> 1, f32 = kind & 1;
        if (count[f32][narrow] == 0) continue;
        split_table(t, f32, narrow, &part);
        lay_out_items(&part, sms);
        const cudaError_t e = launch_table(part, queue, status, blocks_per_sm, clear, stream);
        if (e != cudaSuccess) return e;
        clear = sizeof(unsigned long long);
    }
    return cudaSuccess;
}

}  // namespace dwtfuse
