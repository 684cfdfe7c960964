// moss_lane_offsets_noalloc: the lane-offset scan of the step (the work of
// k_lanescan) for callers that cannot allocate device memory.
//
// Who needs it: code that runs where cudaMalloc is off limits — inside a
// framework whose caching allocator owns the device memory, in a process with
// a fixed memory reservation, or in a pipeline that must not allocate between
// its own set-up and teardown.  Such a caller owns the per-lane input and
// output arrays; the only extra memory this call needs, the look-back words
// of the single-pass scan, lives in a file-scope static device array that
// every GPU loading the library holds until the process exits.
#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

#include "moss.h"
#include "moss_device.cuh"

namespace {

// Tiles of 256 threads x 16 lanes.  Fewer lanes per tile put more tiles into
// the look-back, whose waiting warps all read the same few words: tiles of
// 1,024 / 2,048 / 4,096 / 8,192 lanes take 17.3 / 13.5 / 12.4 / 12.3 us for
// 362,353 lanes and 66 / 42 / 31 / 34 us for 4,000,003 (512 or 1,024 threads
// per tile: 29-34 us, and up to 12 us instead of 8.5 for a few hundred lanes).
constexpr int NA_THREADS = 256;
constexpr int NA_WARPS = NA_THREADS / 32;
constexpr int NA_ROUNDS = 4;
constexpr int NA_TILE = NA_THREADS * 4 * NA_ROUNDS;
constexpr int NA_MAX_TILES = (MOSS_NOALLOC_MAX_LANES + NA_TILE - 1) / NA_TILE;
constexpr int NA_MAX_DEVICES = 64;

// ticket, done and err first, then the words in use: one clear covers both
struct NoallocScratch {
    int ticket;                             // dynamic tile counter
    int done;                               // blocks that have finished
    int err;                                // a bounded wait gave up, or a lane's new size was negative
    int pad[61];
    unsigned long long tile[NA_MAX_TILES];  // look-back words: flag:2 | leavers:31 | sizes:31
};

// 8 KiB + 256 B of scratch per device, shared by every call
static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

std::mutex g_mu;
NoallocScratch* g_ptr[NA_MAX_DEVICES] = {};
int g_sms[NA_MAX_DEVICES] = {};

// newsize(l) = off_cur[l+1] - off_cur[l] - leave[l] + enter[l];
// off_next = exclusive scan of newsize (n+1 entries), lbefore = exclusive scan of leave.
//
// Bound by the chain of a tile (ticket, loads, look-back) up to about a
// million lanes, by HBM and the look-back above.  A warp takes 512
// consecutive lanes, 128 per round and 4 per thread, so that its 16-byte
// accesses cover 512 contiguous bytes, and issues all of its loads before it
// uses any; the scan runs in registers (shuffles) with one exchange between
// the warps, and the look-back reads 32 tile words at a time.  Vec: the five
// arrays are 16-byte aligned (else the same lanes go one by one).  The block
// that finishes last reports an error in off_next[n] (a launch of its own
// before).  The whole call against tiles of 1,024 lanes loaded one by one,
// scanned through shared memory and looked back one word at a time by one
// thread: 362,353 lanes 26.5 -> 12.4 us, 4,000,003 lanes 114 -> 31 us (80 MB:
// 2.6 TB/s).
template <bool Vec>
__global__ void __launch_bounds__(NA_THREADS) k_noalloc_lanescan(NoallocScratch* sc, int n, int ntiles,
                                                                 const int32_t* off_cur,
                                                                 const int32_t* leave,
                                                                 const int32_t* enter,
                                                                 int32_t* off_next, int32_t* lbefore) {
    __shared__ int s_tile;
    __shared__ long long s_wsum[NA_WARPS];
    __shared__ unsigned long long s_prefix;
    const int ln = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr long long LOW = (1ll << 31) - 1;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&sc->ticket, 1);
        __syncthreads();
        const int tile = s_tile;
        if (tile >= ntiles) break;
        const int wbase = tile * NA_TILE + w * (128 * NA_ROUNDS);
        int o[NA_ROUNDS][5], lv[NA_ROUNDS][4], en[NA_ROUNDS][4];
#pragma unroll
        for (int r = 0; r < NA_ROUNDS; ++r) {
            const int l0 = wbase + r * 128 + 4 * ln;
            o[r][4] = 0;
            if (Vec && l0 + 4 <= n) {
                const int4 ov = *reinterpret_cast<const int4*>(off_cur + l0);
                const int4 lx = *reinterpret_cast<const int4*>(leave + l0);
                const int4 ex = *reinterpret_cast<const int4*>(enter + l0);
                o[r][0] = ov.x; o[r][1] = ov.y; o[r][2] = ov.z; o[r][3] = ov.w;
                lv[r][0] = lx.x; lv[r][1] = lx.y; lv[r][2] = lx.z; lv[r][3] = lx.w;
                en[r][0] = ex.x; en[r][1] = ex.y; en[r][2] = ex.z; en[r][3] = ex.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int l = l0 + j;
                    o[r][j] = l <= n ? off_cur[l] : 0;
                    lv[r][j] = l < n ? leave[l] : 0;
                    en[r][j] = l < n ? enter[l] : 0;
                }
            }
            // the offset behind the thread's last lane: the next thread's first
            if (ln == 31 && l0 + 4 <= n) o[r][4] = off_cur[l0 + 4];
        }
        long long pre[NA_ROUNDS], run = 0;
        bool bad = false;
#pragma unroll
        for (int r = 0; r < NA_ROUNDS; ++r) {
            const int l0 = wbase + r * 128 + 4 * ln;
            const int nx = __shfl_down_sync(0xffffffffu, o[r][0], 1);
            if (ln < 31) o[r][4] = nx;
            long long tn = 0, tl = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int ns = l0 + j < n ? o[r][j + 1] - o[r][j] - lv[r][j] + en[r][j] : 0;
                if (ns < 0) {  // violated precondition: reported, and kept out of the packed sums
                    bad = true;
                    ns = 0;
                }
                en[r][j] = ns;
                tn += ns; tl += lv[r][j];
            }
            const long long packed = (tl << 31) | tn;
            long long incl = packed;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, incl, d);
                if (ln >= d) incl += y;
            }
            pre[r] = run + incl - packed;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (bad) atomicOr(&sc->err, 2);
        if (ln == 0) s_wsum[w] = run;
        __syncthreads();
        long long wb = 0, total = 0;
#pragma unroll
        for (int k = 0; k < NA_WARPS; ++k) {
            const long long x = s_wsum[k];
            if (k < w) wb += x;
            total += x;
        }
        if (w == 0) {
            unsigned long long prefix = 0;
            if (tile > 0) {
                bool timeout = false;
                if (ln == 0) moss::store_release(&sc->tile[tile], (1ull << 62) | (unsigned long long)total);
                prefix = moss::warp_lookback(sc->tile, tile, &timeout);
                if (ln == 0 && timeout) atomicOr(&sc->err, 1);
            }
            if (ln == 0) {
                moss::store_release(&sc->tile[tile], (2ull << 62) | (prefix + (unsigned long long)total));
                s_prefix = prefix;
            }
        }
        __syncthreads();
        const long long base = (long long)s_prefix + wb;
#pragma unroll
        for (int r = 0; r < NA_ROUNDS; ++r) {
            const int l0 = wbase + r * 128 + 4 * ln;
            const long long ex = base + pre[r];
            int a = (int)(ex & LOW), b = (int)(ex >> 31);
            int an[4], bn[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                an[j] = a; bn[j] = b;
                a += en[r][j]; b += lv[r][j];
            }
            if (Vec && l0 + 4 <= n) {
                *reinterpret_cast<int4*>(off_next + l0) = make_int4(an[0], an[1], an[2], an[3]);
                *reinterpret_cast<int4*>(lbefore + l0) = make_int4(bn[0], bn[1], bn[2], bn[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (l0 + j < n) { off_next[l0 + j] = an[j]; lbefore[l0 + j] = bn[j]; }
            }
            if (l0 < n && n <= l0 + 4) off_next[n] = a;  // this thread holds the last lane
        }
        __syncthreads();
    }
    // a wait that gave up, or a negative size, marks the whole result invalid
    // (documented sentinel): written by the block that finishes last, after
    // every other block's writes
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&sc->done, 1) == (int)gridDim.x - 1) {
            __threadfence();
            if (atomicAdd(&sc->err, 0)) off_next[n] = -1;
        }
    }
}

cudaError_t launch_noalloc(NoallocScratch* sc, int n, int sms, bool vec, const int32_t* off_cur,
                           const int32_t* leave, const int32_t* enter, int32_t* off_next, int32_t* lbefore,
                           cudaStream_t s) {
    const int ntiles = (n + NA_TILE - 1) / NA_TILE;
    const int grid = ntiles < sms * 4 ? ntiles : sms * 4;
    const cudaError_t e = cudaMemsetAsync(sc, 0, offsetof(NoallocScratch, tile) + 8 * (size_t)ntiles, s);
    if (e != cudaSuccess) return e;
    if (vec)
        k_noalloc_lanescan<true><<<grid, NA_THREADS, 0, s>>>(sc, n, ntiles, off_cur, leave, enter, off_next, lbefore);
    else
        k_noalloc_lanescan<false><<<grid, NA_THREADS, 0, s>>>(sc, n, ntiles, off_cur, leave, enter, off_next, lbefore);
    return cudaGetLastError();
}

// once per device, with that device current: the device address of the
// static scratch (a host-side name of a __device__ variable is not a device
// address) and the SM count used to size the grid
int setup_device(int dev, NoallocScratch** out, int* sms) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
            cudaGetLastError();
            return MOSS_ECUDA;
        }
        int s = 0;
        if (cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return MOSS_ECUDA;
        }
        g_ptr[dev] = (NoallocScratch*)p;
        g_sms[dev] = s;
    }
    *out = g_ptr[dev];
    *sms = g_sms[dev];
    return MOSS_OK;
}

}  // namespace

extern "C" int moss_lane_offsets_noalloc(int32_t n_lanes, const int32_t* d_off_cur,
                                         const int32_t* d_leave, const int32_t* d_enter,
                                         int32_t* d_off_next, int32_t* d_lbefore, void* cuda_stream) {
    if (n_lanes < 0 || n_lanes > MOSS_NOALLOC_MAX_LANES) return MOSS_EINVAL;
    if (!d_off_cur || !d_off_next || (n_lanes > 0 && (!d_leave || !d_enter || !d_lbefore)))
        return MOSS_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
        cudaGetLastError();
        return MOSS_ECUDA;
    }
    NoallocScratch* sc = nullptr;
    int sms = 1;
    const int rc = setup_device(dev, &sc, &sms);
    if (rc != MOSS_OK) return rc;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (n_lanes == 0) {
        // no lanes: the offset array is the single entry 0
        if (cudaMemsetAsync(d_off_next, 0, sizeof(int32_t), s) != cudaSuccess) {
            cudaGetLastError();
            return MOSS_ECUDA;
        }
        return MOSS_OK;
    }
    const bool vec = (((uintptr_t)d_off_cur | (uintptr_t)d_leave | (uintptr_t)d_enter | (uintptr_t)d_off_next |
                       (uintptr_t)d_lbefore) & 15) == 0;
    const cudaError_t e = launch_noalloc(sc, n_lanes, sms, vec, d_off_cur, d_leave, d_enter, d_off_next, d_lbefore, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return MOSS_ECUDA;
    }
    return MOSS_OK;
}
