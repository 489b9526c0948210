// katz_certify_topk_noalloc: certify a top-k ranking from per-node bounds
// without allocating anything.
//
// Some callers cannot let a library call cudaMalloc or cudaFree.  A serving
// process that hands all device memory to its own caching allocator at start
// (PyTorch's, for one) has none left for a library, and must keep every byte
// accounted for in its pool.  A latency-bound loop cannot afford cudaFree,
// which waits for the whole device to go idle and so stalls every other
// stream.  A plug-in host may forbid device allocation by the code it loads.
// For such callers this entry point takes the bounds and the output buffers
// from the caller and keeps its working memory in one file-scope __device__
// array of fixed size, present on every device that loads the library.
//
// Its work is the selection and checking half of an iteration of the
// library's main loop, run over all n nodes:
//   begin    where groups are not needed: every node fits the candidate buffer, or
//            k is above 4096;
//   groups   else: the nodes fall into 8192 groups by a hash of their id; the k-th
//            largest of the groups' largest lower bounds, cut to its upper 22
//            bits, is reached by at least k nodes, and by few more (about 1660
//            for k = 1500, wherever the large bounds lie);
//   compact  the nodes that reach it, the candidates;
//   radix    only when they outgrow the candidate buffer (many equal bounds,
//            k above 4096): a radix select of the k-th 96-bit key, in kernels
//            that return at once otherwise (1 us each; one cooperative kernel
//            instead took 190 us more per call when calls are queued);
//   rank     each candidate's place by counting those before it;
//   cross    the separation of the top-k from each other and from the rest.
// Each of the three passes over the nodes reads one array of 8 n bytes.  A
// radix select over all nodes with a sort in one block took 419 us at n = 4 M,
// k = 1000 (230 of them in global atomics on the few bins that hold most
// bounds); these kernels take 90 us, launches included.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/katz.h"
#include "katz_grid.cuh"

namespace {

using katz::last_block;

constexpr int NA_BINS = 65536;          // 16-bit digits
constexpr int NA_CAP = KATZ_MAX_K;      // candidates held
static_assert((NA_CAP & (NA_CAP - 1)) == 0, "a power of two: places are masked with it");
constexpr int NA_MAX_DEVICES = 64;
constexpr int NA_GROUPS = 8192;
constexpr int NA_GROUP_THREADS = 512;
constexpr int NA_GROUP_BLOCKS = 128;    // 65536 threads, eight for each group
constexpr int NA_GROUP_MAX_K = NA_GROUPS / 2;  // above: more nodes than candidates would reach the k-th group
constexpr int NA_RADIX_THREADS = 512;

struct NoAllocScratch {
    unsigned int hist[NA_BINS];    // radix: histogram; groups: largest bound of each thread; rank: the order
    unsigned int ticket;           // last_block: cleared by every call, zero between its kernels
    int use_radix;
    unsigned int group_key;        // candidates: upper 32 key bits at or above it
    unsigned long long cand_count;
    unsigned long long cross;
    unsigned long long above;      // keys known to lie above the current bucket
    unsigned long long k_rem;      // rank of the k-th key inside the current bucket
    unsigned long long pre_hi;     // selected digits so far (96-bit key: hi 64, lo 32)
    unsigned int pre_lo;
    int done;                      // threshold found
    unsigned long long thr_hi;     // candidates: key >= (thr_hi, thr_lo)
    unsigned int thr_lo;
    int theta_id;                  // k-th node
    unsigned long long theta_key;
    unsigned long long cand_key[NA_CAP];
    double cand_u[NA_CAP];
    int cand_id[NA_CAP];
};

// The working memory of every call on this device (at most 420 KiB).  Calls
// that overlap on the GPU (different streams) race on it.
__device__ __align__(256) NoAllocScratch g_noalloc;

std::mutex g_addr_mu;
NoAllocScratch* g_addr[NA_MAX_DEVICES] = {};
int g_sms[NA_MAX_DEVICES] = {};  // multiprocessors of each device (grid size of the O(n) passes)

typedef unsigned __int128 u128;

// 64-bit key whose unsigned order is the order of the doubles (negative
// values included), then the complemented id: one 96-bit key per node whose
// descending order is (lower bound desc, id asc)
__device__ __forceinline__ unsigned long long order_bits(double l) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(l);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__device__ __forceinline__ double bound_of(unsigned long long key) {  // the inverse
    return __longlong_as_double((long long)((key >> 63) ? key & 0x7fffffffffffffffull : ~key));
}

__device__ __forceinline__ u128 key_of(double l, int v) {
    return ((u128)order_bits(l) << 32) | (u128)(0xffffffffu ^ (unsigned)v);
}

// what a call starts from
__device__ __forceinline__ void begin_call(NoAllocScratch* S, long long k, int use_radix) {
    S->cand_count = 0;
    S->cross = 0;
    S->above = 0;
    S->k_rem = (unsigned long long)k;
    S->pre_hi = 0;
    S->pre_lo = 0;
    S->done = 0;
    S->use_radix = use_radix;
    S->group_key = 0;  // unless the groups give one: every node is taken
}

// the start of a call that needs no groups: every node fits the buffer, or k is
// too large for them
__global__ void na_begin(NoAllocScratch* S, long long k, int use_radix) {
    S->ticket = 0;
    begin_call(S, k, use_radix);
}

// The largest lower bound (upper 32 key bits; 0: no node) of thread t's nodes
// i 65536 + (t ^ mix(i)), i = 0, 1, ...; the last block takes the k-th largest
// over the groups of eight threads s 8192 + (g ^ mix(s)).  Neighbouring large
// bounds (a sorted array) fall into different groups, and so do those of ids
// that differ in a few bits (the hubs of an R-MAT graph: 7700 candidates for k
// = 1000 with groups v mod 8192).  A warp reads whole 256-byte segments.
__device__ __forceinline__ unsigned int mix(unsigned int i) { return (i * 0x9E3779B1u) >> 16; }

__global__ void __launch_bounds__(NA_GROUP_THREADS)
na_groups(NoAllocScratch* S, const double* __restrict__ lower, long long n, long long k) {
    constexpr unsigned int T = NA_GROUP_THREADS * NA_GROUP_BLOCKS;
    static_assert(T == 65536, "mix() gives 16 bits");
    constexpr int U = 16;
    const int tid = threadIdx.x;
    const unsigned int t = blockIdx.x * NA_GROUP_THREADS + tid;
    const unsigned int rounds = (unsigned int)((n + T - 1) / T);
    unsigned int m = 0;
    for (unsigned int i = 0; i < rounds; i += U) {
        double x[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const long long v = (long long)(i + q) * T + (t ^ mix(i + q));
            x[q] = v < n ? __ldg(lower + v) : __longlong_as_double(-1ll);  // key 0: no other is below it, not even a NaN's
        }
#pragma unroll
        for (int q = 0; q < U; ++q) m = max(m, (unsigned int)(order_bits(x[q]) >> 32));
    }
    S->hist[t] = m;
    if (!last_block(&S->ticket)) return;
    if (tid == 0) begin_call(S, k, 0);  // and the key below
    constexpr int PER = NA_GROUPS / NA_GROUP_THREADS;
    unsigned int g[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        unsigned int x = 0;
#pragma unroll
        for (unsigned int s = 0; s < T / NA_GROUPS; ++s)
            x = max(x, __ldcg(&S->hist[s * NA_GROUPS + ((q * NA_GROUP_THREADS + tid) ^ (mix(s) % NA_GROUPS))]));
        g[q] = x;
    }
    // a key that at least k groups reach: the largest one with its lower 10 bits
    // 0 (a mantissa of 10 bits left), two bits a step
    constexpr int STEPS = 11;
    __shared__ int s_cnt[STEPS][3];
    if (tid < 3 * STEPS) (&s_cnt[0][0])[tid] = 0;
    __syncthreads();
    unsigned int key = 0;
    for (int step = 0; step < STEPS; ++step) {
        const int sh = 30 - 2 * step;
        int c[3] = {0, 0, 0};
#pragma unroll
        for (int q = 0; q < PER; ++q)
#pragma unroll
            for (unsigned int d = 0; d < 3; ++d) c[d] += g[q] >= (key | ((d + 1) << sh));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            c[d] = __reduce_add_sync(0xffffffffu, c[d]);
            if ((tid & 31) == 0 && c[d]) atomicAdd(&s_cnt[step][d], c[d]);
        }
        __syncthreads();
        unsigned int d = 3;
        while (d > 0 && s_cnt[step][d - 1] < (int)k) --d;
        key |= d << sh;
    }
    if (tid == 0) S->group_key = key;
}

// a candidate's place in the buffer, one atomic per warp; the buffer keeps the
// first NA_CAP (more: the count says so, and the radix pass starts over).  False
// once the buffer was full before this warp's.
__device__ __forceinline__ bool add_candidate(NoAllocScratch* S, bool take, double l, const double* upper,
                                              long long v) {
    const unsigned m = __ballot_sync(0xffffffffu, take);
    if (!m) return true;
    const int lane = threadIdx.x & 31;
    unsigned long long base = 0;
    if (lane == __ffs(m) - 1) base = atomicAdd(&S->cand_count, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
    const unsigned long long pos = base + __popc(m & ((1u << lane) - 1u));
    if (take && pos < (unsigned long long)NA_CAP) {
        S->cand_key[pos] = order_bits(l);
        S->cand_u[pos] = upper[v];
        S->cand_id[pos] = (int)v;
    }
    return base < (unsigned long long)NA_CAP;
}

__global__ void __launch_bounds__(256)
na_compact(NoAllocScratch* S, const double* __restrict__ lower, const double* __restrict__ upper, long long n) {
    // no counts yet, for the radix select (the groups are done with the array)
    for (int q = blockIdx.x * 256 + threadIdx.x; q < NA_BINS; q += gridDim.x * 256) S->hist[q] = 0;
    if (S->use_radix) return;
    const unsigned int gk = S->group_key;
    constexpr int U = 4;
    const long long tile = 256LL * U;
    for (long long base = (long long)blockIdx.x * tile; base < n; base += gridDim.x * tile) {  // warp-uniform
        double l[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const long long v = base + q * 256 + threadIdx.x;
            l[q] = v < n ? __ldg(lower + v) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const long long v = base + q * 256 + threadIdx.x;
            if (!add_candidate(S, v < n && (unsigned int)(order_bits(l[q]) >> 32) >= gk, l[q], upper, v))
                return;  // the radix select counts them all again
        }
    }
}

__device__ __forceinline__ bool radix_needed(const NoAllocScratch* S) {
    return S->use_radix || S->cand_count > (unsigned long long)NA_CAP;
}

// pick the bucket that holds the k-th key (one block); stop once all keys from
// that bucket up fit the candidate buffer.  A warp sums 128 bins a load, and one
// warp looks through the 128 that hold the key: with a thread per 128 bins, each
// walking its own one load at a time, na_radix of 9000 nodes took 60 us, 11 so.
__device__ void radix_find(NoAllocScratch* S, int pass) {
    constexpr int SLICES = NA_BINS / 128, WARPS = NA_RADIX_THREADS / 32;
    static_assert(SLICES == NA_RADIX_THREADS, "a thread per slice in the scan");
    __shared__ unsigned int part[SLICES], warp_sum[WARPS];  // a digit's counts stay below 2^31
    __shared__ int s_slice, s_bin;
    __shared__ unsigned int s_cum, s_count;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint4* h4 = (const uint4*)S->hist;
    // slice i: the 128 bins from NA_BINS - 128 (i + 1) on; slices count from the top
    auto slice_load = [&](int i, int l) { return __ldcg(h4 + (NA_BINS / 4 - 32 * (i + 1) + l)); };
#pragma unroll 8
    for (int q = 0; q < SLICES / WARPS; ++q) {
        const int i = q * WARPS + wid;
        const uint4 v = slice_load(i, lane);
        const unsigned int sum = __reduce_add_sync(0xffffffffu, v.x + v.y + v.z + v.w);
        if (lane == 0) part[i] = sum;
    }
    if (tid == 0) s_slice = s_bin = -1;
    __syncthreads();
    const unsigned int k = (unsigned int)S->k_rem;
    auto scan = [&](unsigned int x) {  // inclusive, over the lanes
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned int y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        return x;
    };
    const unsigned int mine = part[tid];
    unsigned int upto = scan(mine);
    if (lane == 31) warp_sum[wid] = upto;
    __syncthreads();
    for (int w = 0; w < wid; ++w) upto += warp_sum[w];
    if (upto - mine < k && upto >= k) {
        s_slice = tid;
        s_cum = upto - mine;
    }
    __syncthreads();
    if (wid == 0 && s_slice >= 0) {
        const uint4 v = slice_load(s_slice, 31 - lane);  // lane 0: the top four bins, w the first
        const unsigned int before = s_cum;
        const unsigned int four = v.x + v.y + v.z + v.w, in = before + scan(four);
        unsigned int cum = in - four;
        if (cum < k && in >= k) {
            const unsigned int h[4] = {v.w, v.z, v.y, v.x};
            int q = 0;
            while (cum + h[q] < k) cum += h[q++];
            s_bin = NA_BINS - 1 - 128 * s_slice - 4 * lane - q;
            s_count = h[q];
            s_cum = cum;
        }
    }
    __syncthreads();
    const int b = s_bin;
    const unsigned long long hb = s_count, cum_sel = s_cum;
    for (int q = tid; q < NA_BINS / 4; q += NA_RADIX_THREADS)  // ready for the next pass
        ((uint4*)S->hist)[q] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0 && b >= 0) {
        const int shift = 80 - 16 * pass;
        const u128 pre = (((u128)S->pre_hi << 32) | S->pre_lo) | ((u128)(unsigned)b << shift);
        const unsigned long long above = S->above + cum_sel;
        if (above + hb <= (unsigned long long)NA_CAP || pass == 5) {
            S->done = 1;
            S->thr_hi = (unsigned long long)(pre >> 32);
            S->thr_lo = (unsigned int)pre;
            S->cand_count = 0;  // na_radix_compact counts again
        } else {
            S->above = above;
            S->k_rem = k - cum_sel;
            S->pre_hi = (unsigned long long)(pre >> 32);
            S->pre_lo = (unsigned int)pre;
        }
    }
}

// histogram of digit `pass` (bits 95-16*pass .. 80-16*pass) of the keys that
// share the digits chosen so far; the lanes of a warp that hit the same bin
// (bounds of one magnitude share their top digits) add once.  The last block
// picks the bucket.
__global__ void __launch_bounds__(NA_RADIX_THREADS)
na_radix(NoAllocScratch* S, const double* __restrict__ lower, long long n, int pass) {
    if (!radix_needed(S) || S->done) return;
    const int shift = 80 - 16 * pass;
    const u128 pre = ((u128)S->pre_hi << 32) | S->pre_lo;
    const int lane = threadIdx.x & 31;
    // base is the same for every thread of a block, so the loop is warp-uniform
    for (long long base = (long long)blockIdx.x * blockDim.x; base < n; base += (long long)gridDim.x * blockDim.x) {
        const long long v = base + threadIdx.x;
        unsigned bin = 0x10000u;  // none
        if (v < n) {
            const u128 key = key_of(lower[v], (int)v);
            if (pass == 0 || (key >> (shift + 16)) == (pre >> (shift + 16))) bin = (unsigned)(key >> shift) & 0xffffu;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, bin);
        if (bin < 0x10000u && lane == __ffs(peers) - 1) atomicAdd(&S->hist[bin], (unsigned)__popc(peers));
    }
    if (last_block(&S->ticket)) radix_find(S, pass);
}

// after the last pass: the candidates at or above the threshold
__global__ void __launch_bounds__(256)
na_radix_compact(NoAllocScratch* S, const double* __restrict__ lower, const double* __restrict__ upper, long long n) {
    if (!S->done) return;
    const u128 thr = ((u128)S->thr_hi << 32) | S->thr_lo;
    for (long long base = (long long)blockIdx.x * 256; base < n; base += (long long)gridDim.x * 256) {
        const long long v = base + threadIdx.x;
        const double l = v < n ? lower[v] : 0.0;
        add_candidate(S, v < n && key_of(l, (int)v) >= thr, l, upper, v);
    }
}

// the candidates' places in the order (lower desc, id asc): the first k are
// the ranking (and the order that na_cross checks), the k-th gives theta
__global__ void __launch_bounds__(katz::RANK_THREADS) na_rank(NoAllocScratch* S, long long k, int32_t* ids_out) {
    const int cnt = (int)min((unsigned long long)NA_CAP, S->cand_count);
    // i0 is the same for every thread of a block
    for (int i0 = blockIdx.x * katz::RANK_PER_BLOCK; i0 < cnt; i0 += gridDim.x * katz::RANK_PER_BLOCK) {
        const int i = i0 + threadIdx.x / katz::RANK_LANES;
        const unsigned long long key = i < cnt ? S->cand_key[i] : 0ull;
        const int id = i < cnt ? S->cand_id[i] : 0x7fffffff;
        const int r = katz::rank_by_count(S->cand_key, S->cand_id, cnt, key, id);
        if (i < cnt && r < k && threadIdx.x % katz::RANK_LANES == 0) {
            ids_out[r] = id;
            S->hist[r] = (unsigned int)i;
            if (r == k - 1) {
                S->theta_key = key;
                S->theta_id = id;
            }
        }
    }
}

// the candidate that a word of the order names: within the candidate arrays
// whatever an overlapping call wrote there
__host__ __device__ constexpr unsigned int place_of(unsigned int word) { return word & (NA_CAP - 1u); }

// every node outside the top-k must be eps-separated from the k-th (only the
// nodes whose upper bound reaches theta need their lower bound looked at),
// and adjacent top-k pairs from each other; the last block gives the verdict
__global__ void __launch_bounds__(256)
na_cross(NoAllocScratch* S, const double* __restrict__ lower, const double* __restrict__ upper, long long n,
         long long k, double eps, int32_t* certified_out) {
    const double th = bound_of(S->theta_key);
    const unsigned long long th_bits = S->theta_key;
    const u128 th_key = ((u128)th_bits << 32) | (u128)(0xffffffffu ^ (unsigned)S->theta_id);
    unsigned long long c = 0;
    constexpr int U = 4;
    const long long tile = 256LL * U;
    for (long long base = (long long)blockIdx.x * tile; base < n; base += gridDim.x * tile) {
        double u[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const long long v = base + q * 256 + threadIdx.x;
            u[q] = v < n ? __ldg(upper + v) : 0.0;
        }
        // u - eps >= theta needs u >= theta (eps > 0): an integer compare first;
        // the FP64 pipe (narrow on this GPU: it took 20 us here) sees only the
        // warps with a node that passes
        bool near = false;
#pragma unroll
        for (int q = 0; q < U; ++q) near |= order_bits(u[q]) >= th_bits;
        if (!__any_sync(0xffffffffu, near)) continue;
        for (int q = 0; q < U; ++q) {
            const long long v = base + q * 256 + threadIdx.x;
            if (v < n && __dsub_rn(u[q], eps) >= th && key_of(lower[v], (int)v) < th_key) ++c;
        }
    }
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
    for (long long r = t + 1; r < k; r += (long long)gridDim.x * 256)
        if (__dsub_rn(S->cand_u[place_of(S->hist[r])], eps) >= bound_of(S->cand_key[place_of(S->hist[r - 1])])) ++c;
    for (int off = 16; off; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&S->cross, c);
    if (last_block(&S->ticket) && threadIdx.x == 0)
        *certified_out = __ldcg(&S->cross) == 0;
}

// Address of the scratch array on the current device and the device's
// multiprocessor count, resolved once per device.
katz_status scratch_on_current_device(NoAllocScratch** out, int* sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return KATZ_ECUDA;
    std::lock_guard<std::mutex> lock(g_addr_mu);
    if (!g_addr[dev]) {
        void* p = nullptr;
        int count = 0;
        if (cudaGetSymbolAddress(&p, g_noalloc) != cudaSuccess) return KATZ_ECUDA;
        if (cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || count < 1)
            return KATZ_ECUDA;
        g_sms[dev] = count;
        g_addr[dev] = (NoAllocScratch*)p;
    }
    *out = g_addr[dev];
    *sms = g_sms[dev];
    return KATZ_OK;
}

}  // namespace

extern "C" katz_status katz_certify_topk_noalloc(const double* lower, const double* upper, int64_t n, int64_t k,
                                                 double eps, int32_t* ids_out, int32_t* certified_out,
                                                 void* cuda_stream) {
    if (!lower || !upper || !ids_out || !certified_out) return KATZ_EINVAL;
    if (n < 1 || n > 0x7ffffffeLL || k < 1 || k > n || k > KATZ_MAX_K || !(eps > 0.0)) return KATZ_EINVAL;
    static_assert(sizeof(NoAllocScratch) <= 420 * 1024, "the stated size of the array");
    // an error left by the caller's earlier work stays the caller's: it is
    // neither cleared here nor reported as a failure of this call's launches
    if (cudaPeekAtLastError() != cudaSuccess) return KATZ_ECUDA;
    NoAllocScratch* S = nullptr;
    int sms = 0;
    katz_status st = scratch_on_current_device(&S, &sms);
    if (st != KATZ_OK) return st;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const long long nn = (long long)n, kk = (long long)k;
    const long long cap = 8LL * sms;  // eight 256-thread blocks per multiprocessor, grid-stride beyond
    const int grid = (int)((n + 1023) / 1024 < cap ? (n + 1023) / 1024 : cap);
    // either start clears the count of finished blocks: calls that overlapped may
    // have left one behind, which would make every later call wrong
    if (n <= NA_CAP || k > NA_GROUP_MAX_K) {
        na_begin<<<1, 1, 0, s>>>(S, kk, n > NA_CAP);
    } else {
        if (cudaMemsetAsync(&S->ticket, 0, sizeof(S->ticket), s) != cudaSuccess) {
            cudaGetLastError();
            return KATZ_ECUDA;
        }
        na_groups<<<NA_GROUP_BLOCKS, NA_GROUP_THREADS, 0, s>>>(S, lower, nn, kk);
    }
    na_compact<<<grid, 256, 0, s>>>(S, lower, upper, nn);
    if (n > NA_CAP) {  // else every node fits
        const int rgrid = (int)((n + NA_RADIX_THREADS - 1) / NA_RADIX_THREADS < cap / 2
                                    ? (n + NA_RADIX_THREADS - 1) / NA_RADIX_THREADS : cap / 2);
        for (int pass = 0; pass < 6; ++pass) na_radix<<<rgrid, NA_RADIX_THREADS, 0, s>>>(S, lower, nn, pass);
        na_radix_compact<<<grid, 256, 0, s>>>(S, lower, upper, nn);
    }
    na_rank<<<NA_CAP / katz::RANK_PER_BLOCK, katz::RANK_THREADS, 0, s>>>(S, kk, ids_out);
    na_cross<<<grid, 256, 0, s>>>(S, lower, upper, nn, kk, eps, certified_out);
    return cudaGetLastError() == cudaSuccess ? KATZ_OK : KATZ_ECUDA;
}
