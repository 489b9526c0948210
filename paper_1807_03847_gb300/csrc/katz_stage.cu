// Staged gathers for walk vectors far larger than L2.
//
// A gather of s_{r-1} that misses L2 moves a whole 128-byte line from DRAM for
// 8 bytes: on a Chung-Lu graph of 2^27 vertices a level read 111 GB against 14
// GB of algorithmic bytes, at the measured copy bandwidth.  So the arcs into
// the cold part of the vector (internal ids from `hot` on: the low-degree end
// of the degree-class order) get their values in two steps that only stream:
//
//   1. stage_gather: the cold part is cut into windows of STAGE_WIN entries.
//      A block loads one window into shared memory and writes, for every arc
//      into it, the value gathered there to the arc's place in y.  The rows
//      form STAGE_BANDS runs of equal numbers of arcs; y holds one band after
//      the other, and in a band the places of one window's arcs are
//      consecutive, in the order of the arcs' rows (a segment).
//   2. the SpMV reads y at the arc's place instead of the vector.  Rows that
//      run at the same time take neighbouring places of every window, so each
//      line of y is fetched once and shared while it is in L2, and the places
//      in use at one time lie in one band.  With y in one band
//      (7.6 GB at 2^27 vertices, one page of every window in use at a time) the
//      SpMV took 16.3 ms; address translation bound it, not DRAM (24 GB read).
//      32 bands: 9.7 ms; 16 bands: 13.6 for the level in place of 11.6.
//
// Per cold arc that is 2 + 8 bytes in step 1 and 8 in step 2 (4-byte values: 2
// + 4 and 4) in place of 128.  The values and the order of every row sum are
// those of the plain gather, so the results are the same bits.
//
// Measured on that graph, FP64: a level 17.1 -> 11.4 ms when it came, 10.6 now with
// fewer rows per warp (1.8 of it step 1; 37.4 GB read and 7.8 written by both
// steps).  Rankings before it and now, the SpMV's row batches included: 185 -> 121
// ms; Chung-Lu n = 6e7: 64.7 -> 48.6, FP32-certified 59.4 -> 47.6; n = 4e7: 39.1 ->
// 32.0; G(3.6e7, 4 n): 50.3 -> 27.9.  Building it takes no more of a create than the
// anchor order (katz_relabel.cu), which it replaces: 59 against 75 ms at 2^27.
// Below 2^25 vertices the gain (2.68 -> 2.54 ms a level at 2^25 - 39) does not pay
// for a create three times as long.
//
// 2^23 hot entries, 8192 per window: against 11.4 ms a level then, 2^22 took 11.6 ms,
// 2^21 12.5, 2^24 12.3 (the hot part contends for L2); 64 or 128 bands changed
// nothing; windows of 16384 (one block per SM) 16.1 ms with 16 bands.
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "katz_common.cuh"
#include "katz_handle.h"

namespace katz {

namespace {

constexpr int STAGE_BITS = 13;
constexpr int STAGE_WIN = 1 << STAGE_BITS;   // entries per window: 64 KB of FP64, three blocks per SM
constexpr int STAGE_THREADS = 512;
constexpr int STAGE_WARPS = STAGE_THREADS / 32;
constexpr int STAGE_BANDS = 2 * STAGE_WARPS; // runs of rows with equal numbers of arcs
constexpr int STAGE_CHUNK = 1 << 16;         // arcs per block: a window is loaded once per chunk
constexpr int STAGE_ALIGN = 32;              // places of a segment start at a multiple of this
constexpr int STAGE_MAX_WINDOWS = 1 << 15;   // 128 KB of counters in shared memory
constexpr int STAGE_HIST_BLOCKS = 10;        // per band
constexpr int STAGE_ASSIGN = 2048;           // arcs per block of the assignment; a band is a multiple of it
constexpr int STAGE_CACHED = 1024;           // windows that a plain gather may find in L2 (64 MB of FP64)
constexpr int STAGE_RUNS = 64;               // sampled runs per band, of STAGE_RUN arcs each
constexpr int STAGE_RUN = 1024;

int64_t stage_windows(int64_t n) { return (n - STAGE_HOT + STAGE_WIN - 1) / STAGE_WIN; }

int64_t stage_band_arcs(int64_t nnz) {
    return ((nnz + STAGE_BANDS - 1) / STAGE_BANDS + STAGE_ASSIGN - 1) / STAGE_ASSIGN * STAGE_ASSIGN;
}

// A sample of the arcs of one band (a block): out[0] += its cold arcs, out[1] +=
// those outside the STAGE_CACHED windows of the vector that the band uses most.
__global__ void __launch_bounds__(STAGE_RUN)
stage_sample_kernel(const int32_t* __restrict__ col, int64_t nnz, int64_t band_arcs, int hot_windows, int windows,
                    unsigned long long* out) {
    extern __shared__ unsigned int h[];
    __shared__ unsigned int s_cold, s_above, s_held;
    const int tid = threadIdx.x, lane = tid & 31;
    for (int q = tid; q < windows; q += STAGE_RUN) h[q] = 0;
    if (tid == 0) s_cold = 0;
    __syncthreads();
    const int64_t begin = blockIdx.x * band_arcs, end = min(nnz, begin + band_arcs);
    const int64_t step = max((end - begin) / STAGE_RUNS, (int64_t)STAGE_RUN);
    unsigned int cold = 0;
#pragma unroll 8
    for (int r = 0; r < STAGE_RUNS; ++r) {
        const int64_t j = begin + r * step + tid;
        const int w = j < end ? col[j] >> STAGE_BITS : -1;
        // lanes of one window add once: near neighbours share theirs
        const unsigned peers = __match_any_sync(0xffffffffu, w);
        if (w >= 0 && lane == __ffs(peers) - 1) atomicAdd(&h[w], (unsigned)__popc(peers));
        cold += w >= hot_windows;
    }
    cold = __reduce_add_sync(0xffffffffu, cold);
    if (lane == 0) atomicAdd(&s_cold, cold);
    // the smallest count that at most STAGE_CACHED windows exceed, and the cold
    // arcs of the windows that do
    unsigned int lo = 0, hi = STAGE_RUNS * STAGE_RUN;
    for (bool last = false;; last = lo == hi) {
        if (tid == 0) s_above = s_held = 0;
        __syncthreads();
        const unsigned int mid = (lo + hi) / 2;
        unsigned int above = 0, held = 0;
        for (int q = tid; q < windows; q += STAGE_RUN)
            if (h[q] > mid) {
                ++above;
                held += q >= hot_windows ? h[q] : 0u;
            }
        above = __reduce_add_sync(0xffffffffu, above);
        held = __reduce_add_sync(0xffffffffu, held);
        if (lane == 0) {
            atomicAdd(&s_above, above);
            atomicAdd(&s_held, held);
        }
        __syncthreads();
        above = s_above;
        __syncthreads();  // read before the next round's zeroes
        if (last) break;
        if (above <= STAGE_CACHED) hi = mid;
        else lo = mid + 1;
    }
    if (tid == 0 && s_cold) {
        atomicAdd(&out[0], s_cold);
        atomicAdd(&out[1], s_cold - s_held);
    }
}

// arcs of every band into every window (gridDim.y: the band)
__global__ void __launch_bounds__(1024)
stage_hist_kernel(const int32_t* __restrict__ col, int64_t nnz, int64_t band_arcs, uint32_t hot, int windows,
                  unsigned int* counts) {
    extern __shared__ unsigned int h[];
    for (int q = threadIdx.x; q < windows; q += blockDim.x) h[q] = 0;
    __syncthreads();
    const int64_t end = min(nnz, (int64_t)(blockIdx.y + 1) * band_arcs);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j0 = blockIdx.y * band_arcs + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j0 < end;
         j0 += 4 * stride) {
        uint32_t c[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = j0 + q * stride < end ? (uint32_t)col[j0 + q * stride] : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (c[q] >= hot) atomicAdd(&h[(c[q] - hot) >> STAGE_BITS], 1u);
    }
    __syncthreads();
    unsigned int* out = counts + (size_t)blockIdx.y * windows;
    for (int q = threadIdx.x; q < windows; q += blockDim.x)
        if (h[q]) atomicAdd(&out[q], h[q]);
}

// the place of every cold arc: blocks run in arc order, so the places of a
// segment follow the order of the rows up to the blocks in flight
__global__ void __launch_bounds__(256)
stage_assign_kernel(const int32_t* __restrict__ col, int64_t nnz, int64_t band_arcs, uint32_t hot, int windows,
                    unsigned int* cursor, uint32_t* __restrict__ src, uint16_t* __restrict__ local) {
    const int64_t j0 = (int64_t)blockIdx.x * STAGE_ASSIGN + threadIdx.x;
    unsigned int* cur = cursor + (size_t)((int64_t)blockIdx.x * STAGE_ASSIGN / band_arcs) * windows;
    constexpr int U = STAGE_ASSIGN / 256;
    uint32_t c[U], p[U];
#pragma unroll
    for (int q = 0; q < U; ++q) c[q] = j0 + q * 256 < nnz ? (uint32_t)col[j0 + q * 256] : 0u;
#pragma unroll
    for (int q = 0; q < U; ++q) p[q] = c[q] >= hot ? atomicAdd(&cur[(c[q] - hot) >> STAGE_BITS], 1u) : 0u;
#pragma unroll
    for (int q = 0; q < U; ++q) {
        if (j0 + q * 256 >= nnz) continue;
        if (c[q] >= hot) local[p[q]] = (uint16_t)((c[q] - hot) & (STAGE_WIN - 1));
        src[j0 + q * 256] = c[q] >= hot ? hot + p[q] : c[q];
    }
}

// y[p] = x[entry of place p] for the places of one window in some bands, a
// warp per band
template <typename T>
__device__ __forceinline__ void stage_window(const T* __restrict__ x, int64_t n, const StageMap& m,
                                             const StageItem& it, T* win) {
    const int64_t base = (int64_t)m.hot + ((int64_t)it.window << STAGE_BITS);
    const int len = (int)min((int64_t)STAGE_WIN, n - base);
    constexpr int V = 16 / (int)sizeof(T);
    const uint4* __restrict__ src = (const uint4*)(x + base);  // 16-byte aligned: base and the slots are
#pragma unroll 4
    for (int q = threadIdx.x; q < len / V; q += STAGE_THREADS) ((uint4*)win)[q] = src[q];
    for (int q = len / V * V + threadIdx.x; q < len; q += STAGE_THREADS) win[q] = x[base + q];
    __syncthreads();
    // two places per lane (a place past a segment's last one holds entry 0 and is read by no arc)
    struct alignas(2 * sizeof(T)) Two { T a, b; };
    const int lane = threadIdx.x & 31;
    for (int band = it.band0 + (threadIdx.x >> 5); band < it.band1; band += STAGE_WARPS) {
        const uint32_t first = m.first[(size_t)band * m.windows + it.window];
        const int pairs = (int)(m.first[(size_t)band * m.windows + it.window + 1] - first) / 2;  // padded
        const ushort2* __restrict__ l2 = (const ushort2*)(m.local + first);
        Two* __restrict__ y2 = (Two*)((T*)m.y + first);
#pragma unroll 4
        for (int q = lane; q < pairs; q += 32) {
            const ushort2 e = __ldcs(l2 + q);
            y2[q] = Two{win[e.x], win[e.y]};
        }
    }
}

// level types as in spmv_rows_kernel: the FP64 slot, the roundings s32, or the
// FP32 slot of level r-1
__global__ void __launch_bounds__(STAGE_THREADS, 3)
stage_gather_kernel(StageMap m, const double* walk, const float* __restrict__ s32, const Ctrl* ctrl, IterParams p) {
    extern __shared__ uint4 win[];
    if (ctrl->stop) return;
    const int r_cur = ctrl->r + 1, f32_from = ctrl->f32_from;
    const double* xs = walk_slot(walk, p, r_cur - 1);
    const StageItem it = m.items[blockIdx.x];
    if (r_cur < f32_from)
        stage_window<double>(xs, p.n, m, it, (double*)win);
    else
        stage_window<float>(r_cur == f32_from ? s32 : (const float*)xs, p.n, m, it, (float*)win);
}

}  // namespace

cudaError_t launch_stage(const DeviceGraph& g, const IterBuffers& b, const IterParams& p, cudaStream_t st) {
    stage_gather_kernel<<<(unsigned)g.stage.n_items, STAGE_THREADS, STAGE_WIN * sizeof(double), st>>>(
        g.stage, (const double*)b.walk, b.s32, b.ctrl, p);
    return cudaGetLastError();
}

void stage_free(katz_handle* h) {
    StageMap& m = h->g.stage;
    dfree(h, m.src);
    dfree(h, m.local);
    dfree(h, m.y);
    dfree(h, m.items);
    dfree(h, m.first);
    m = StageMap();
}

// Worth it where many arcs are cold.  In a symmetric graph as many arcs lead
// into the rows from STAGE_HOT on as leave them; for a directed one that is an
// estimate.  The places must fit 32 bits and the windows' counters one block.
static bool stage_wanted(const katz_handle* h, int64_t head_arcs) {
    const int64_t n = h->g.n, nnz = h->g.nnz, cold = nnz - head_arcs;
    if (n < STAGE_MIN_N || h->opts.keep_history || cold < nnz / 8) return false;
    const int64_t windows = stage_windows(n);
    return windows <= STAGE_MAX_WINDOWS &&
           STAGE_HOT + cold + windows * STAGE_BANDS * STAGE_ALIGN <= (int64_t)0xffffffff;
}

// Whether the graph's gathers would miss: of a sample of the cold arcs, three
// in ten or more lie outside the windows that their band uses most, as many as
// half of L2 holds.  Where ids are near their neighbours' (rings, grids, banded
// matrices) plain gathers hit, and a window's arcs all come from one band, so
// that one warp does their staging and every arc's place comes from one counter.
// At n = 2^25 + 11, 8 arcs a row (three in four of them cold), by the share of
// sampled cold arcs that miss: us a level with plain gathers, with staged ones:
//   ring 0: 735, 4058    grid 0: 633, 2228    neighbours within 2^20 .03: 1231,
//   2636    2^22 .11: 1623, 1985    6 x 2^20 .37: 2250, 1787    2^24 .84: 3113,
//   1707    ring with a tenth of its edges random .06: 1101, 3520    three tenths
//   .22: 1954, 2832    half .40: 2603, 2374    seven tenths .58: 2936, 2069
// G(n, m) and Chung-Lu graphs have shares of .76 to .92.  The creates of the
// ring and the grid: 8.0 and 6.9 ms plain, 98 and 28 staged.  The sample reads
// 2 M arcs.
cudaError_t stage_pays(katz_handle* h, int64_t head_arcs, bool* pays) {
    *pays = false;
    if (!stage_wanted(h, head_arcs)) return cudaSuccess;
    constexpr int hot_windows = (int)(STAGE_HOT / STAGE_WIN);
    const int windows = hot_windows + (int)stage_windows(h->g.n);
    unsigned long long* sums = nullptr;
    unsigned long long* out = (unsigned long long*)(h->h_small + H_SMALL - 16);
    cudaError_t e = dmalloc(h, &sums, 2);
    if (e != cudaSuccess) {  // no memory: plain gathers
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? cudaSuccess : e;
    }
    e = cudaMemsetAsync(sums, 0, 2 * sizeof(unsigned long long), h->stream);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(stage_sample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (hot_windows + STAGE_MAX_WINDOWS) * (int)sizeof(unsigned int));
    if (e == cudaSuccess) {
        stage_sample_kernel<<<STAGE_BANDS, STAGE_RUN, (size_t)windows * sizeof(unsigned int), h->stream>>>(
            h->g.col, h->g.nnz, stage_band_arcs(h->g.nnz), hot_windows, windows, sums);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(out, sums, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    dfree(h, sums);
    if (e == cudaSuccess) *pays = out[0] > 0 && 10 * out[1] >= 3 * out[0];
    return e;
}

// The staged gathers of the graph a handle holds (its final internal order).
// Without the memory for them the handle goes on with plain gathers.  Waits
// for the handle's stream.
cudaError_t stage_build(katz_handle* h) {
    DeviceGraph& g = h->g;
    const uint32_t hot = (uint32_t)STAGE_HOT;
    const int64_t windows = stage_windows(g.n);
    cudaError_t e;
    const size_t cells = (size_t)windows * STAGE_BANDS;
    const int64_t band_arcs = stage_band_arcs(g.nnz);
    unsigned int* counts = nullptr;
    if ((e = dmalloc(h, &counts, cells)) != cudaSuccess) {
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? cudaSuccess : e;
    }
    std::vector<unsigned int> cnt(cells), first(cells + 1);
    e = cudaMemsetAsync(counts, 0, cells * sizeof(unsigned int), h->stream);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(stage_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 STAGE_MAX_WINDOWS * (int)sizeof(unsigned int));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(stage_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 STAGE_WIN * (int)sizeof(double));
    if (e == cudaSuccess) {
        stage_hist_kernel<<<dim3(STAGE_HIST_BLOCKS, STAGE_BANDS), 1024, (size_t)windows * sizeof(unsigned int),
                            h->stream>>>(g.col, g.nnz, band_arcs, hot, (int)windows, counts);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(cnt.data(), counts, cells * sizeof(unsigned int), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) {
        dfree(h, counts);
        return e;
    }
    int64_t places = 0;
    for (size_t q = 0; q < cells; ++q) {
        first[q] = (unsigned int)places;
        places += ((int64_t)cnt[q] + STAGE_ALIGN - 1) / STAGE_ALIGN * STAGE_ALIGN;
    }
    first[cells] = (unsigned int)places;
    if (places == 0 || places + STAGE_HOT > 0xffffffffll) {
        dfree(h, counts);
        return cudaSuccess;
    }
    std::vector<StageItem> items;
    for (int64_t w = 0; w < windows; ++w) {
        int64_t arcs = 0;
        int band0 = 0;
        for (int band = 0; band < STAGE_BANDS; ++band) {
            arcs += cnt[(size_t)band * windows + w];
            if (arcs >= STAGE_CHUNK || band + 1 == STAGE_BANDS) {
                if (arcs > 0) items.push_back(StageItem{(int32_t)w, band0, band + 1});
                arcs = 0;
                band0 = band + 1;
            }
        }
    }
    // at most a quarter of the memory left, the library's own free blocks
    // included: a ranking's buffers and the caller's work come first
    size_t free_b = 0, total_b = 0;
    unsigned long long reserved = 0, used = 0;
    const cudaMemPool_t pool = library_pool(h->dev);
    if ((e = cudaMemGetInfo(&free_b, &total_b)) == cudaSuccess &&
        (e = cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved)) == cudaSuccess)
        e = cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used);
    const double need = 4.0 * (double)g.nnz + 10.0 * (double)places + 4.0 * (double)cells;
    if (e != cudaSuccess || need > 0.25 * ((double)free_b + (double)(reserved - used))) {
        dfree(h, counts);
        return e;
    }
    StageMap& m = g.stage;
    if ((e = dmalloc(h, &m.src, (size_t)g.nnz)) == cudaSuccess &&
        (e = dmalloc(h, &m.local, (size_t)places)) == cudaSuccess &&
        (e = dmalloc(h, (double**)&m.y, (size_t)places)) == cudaSuccess &&
        (e = dmalloc(h, &m.first, cells + 1)) == cudaSuccess)
        e = dmalloc(h, &m.items, items.size());
    if (e != cudaSuccess) {  // no memory: plain gathers
        cudaGetLastError();
        dfree(h, counts);
        stage_free(h);
        return e == cudaErrorMemoryAllocation ? cudaSuccess : e;
    }
    e = cudaMemcpyAsync(m.first, first.data(), (cells + 1) * sizeof(unsigned int), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(counts, m.first, cells * sizeof(unsigned int), cudaMemcpyDeviceToDevice, h->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m.items, items.data(), items.size() * sizeof(StageItem), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m.local, 0, (size_t)places * sizeof(uint16_t), h->stream);
    if (e == cudaSuccess) {
        stage_assign_kernel<<<(unsigned)((g.nnz + STAGE_ASSIGN - 1) / STAGE_ASSIGN), 256, 0, h->stream>>>(
            g.col, g.nnz, band_arcs, hot, (int)windows, counts, m.src, m.local);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);  // the host arrays above are in use until here
    dfree(h, counts);
    if (e != cudaSuccess) {
        stage_free(h);
        return e;
    }
    m.n_items = (int32_t)items.size();
    m.windows = (int32_t)windows;
    m.hot = hot;
    // fewer rows per warp: the rows in flight reach over less of every band (2^27
    // vertices: 11.3 ms a level with four passes, 10.5 with one and four, 10.4 so)
    const SpmvLayout L = g.layout;
    g.layout = make_layout(L.n, L.row_warp, L.row_octet, L.row_thread, L.chunks, 1, 2);
    g.layout.row_empty = L.row_empty;
    return cudaSuccess;
}

}  // namespace katz
