// ts_prims.cu -- device primitives: exclusive scans and a stable LSD radix sort.
//
// Index building sorts segment keys and turns bin counts into offset arrays (radix sort plus
// prefix sums, the GB300 form of the paper's sorted arrays and bin ranges, Sec. 4.1-4.3); the
// search scans per-tile hit counts into output offsets. All of it is hand-written here.
#include <stdarg.h>
#include <stdio.h>

#include <atomic>

#include <algorithm>
#include <mutex>

#include "ts_internal.cuh"

namespace ts {

// ---------------------------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------------------------
static thread_local char g_err[512] = "";
static std::atomic<unsigned long long> g_launches{0};

void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
void note_launches(unsigned long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
unsigned long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

void set_error(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

const char *last_error() { return g_err; }

ts_status cuda_status(cudaError_t e, const char *what)
{
    if (e == cudaErrorMemoryAllocation) {
        set_error("out of device memory in %s", what);
        cudaGetLastError();
        return TS_ERR_OOM;
    }
    set_error("CUDA error in %s: %s", what, cudaGetErrorString(e));
    return TS_ERR_CUDA;
}

void DevBuf::release()
{
    if (p) cudaFreeAsync(p, s);
    p = nullptr;
    bytes = 0;
}

// The library's stream-ordered pools of a device, one for work buffers and rows and one for the
// indexes' arrays: freed blocks stay in the pool (no release threshold), so the work buffers of
// repeated searches, and the arrays of indexes built one after another, are not mapped and
// unmapped every call. (Two, so that what freed indexes leave can be bounded by itself.)
static cudaMemPool_t device_pool(bool index)
{
    static std::mutex mu;
    static cudaMemPool_t pools[64][2] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    cudaMemPool_t &pool = pools[dev][index ? 1 : 0];
    if (!pool) {
        cudaMemPoolProps props;
        memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
            cudaGetLastError();
            pool = nullptr;
            return nullptr;
        }
        uint64_t keep = ~0ull;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    return pool;
}

void pool_trim()
{
    cudaMemPool_t work = device_pool(false), index = device_pool(true);
    if (cudaDeviceSynchronize() == cudaSuccess) {
        if (work) cudaMemPoolTrimTo(work, 0);
        if (index) cudaMemPoolTrimTo(index, 0);
    }
    cudaGetLastError();
}

// Allocations of this thread until the ones that a test lets fail, and how many those are.
static thread_local uint64_t g_fail_after = 0, g_fail_count = 0;

void fail_allocs(uint64_t after, uint64_t count)
{
    g_fail_after = after;
    g_fail_count = count;
}

cudaError_t pool_malloc(void **p, size_t nbytes, cudaStream_t stream, bool index)
{
    if (g_fail_count) {
        if (g_fail_after) {
            g_fail_after--;
        } else {
            g_fail_count--;
            *p = nullptr;
            return cudaErrorMemoryAllocation;
        }
    }
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(stream, &cs);
    cudaMemPool_t pool = cs == cudaStreamCaptureStatusNone ? device_pool(index) : nullptr;
    return pool ? cudaMallocFromPoolAsync(p, nbytes, pool, stream)
                : cudaMallocAsync(p, nbytes, stream);
}

// Bytes of the indexes alive on a device, and the most that the pool holds for them. (Counted here:
// the pool's own count of used memory leaves out what cudaFree gave back.)
struct IndexBytes {
    std::mutex mu;
    uint64_t live = 0, held = 0;
};
static IndexBytes g_index_bytes[64];

cudaError_t index_malloc(void **p, size_t nbytes, cudaStream_t stream, int device)
{
    const cudaError_t e = pool_malloc(p, nbytes, stream, true);
    if (e == cudaSuccess && device >= 0 && device < 64) {
        IndexBytes &b = g_index_bytes[device];
        std::lock_guard<std::mutex> lk(b.mu);
        b.live += nbytes;
        b.held = std::max(b.held, b.live);
    }
    return e;
}

void index_free(void *const *p, size_t n, size_t bytes, size_t keep, int device)
{
    for (size_t k = 0; k < n; k++) cudaFree(p[k]);
    if (device < 0 || device >= 64) return;
    IndexBytes &b = g_index_bytes[device];
    std::lock_guard<std::mutex> lk(b.mu);
    b.live -= bytes;
    if (b.held <= b.live + keep) return;
    b.held = b.live + keep;
    // (given back in whole blocks, and only what a wait has seen freed)
    cudaMemPool_t pool = device_pool(true);
    if (pool && cudaDeviceSynchronize() == cudaSuccess) cudaMemPoolTrimTo(pool, b.held);
    cudaGetLastError();
}

ts_status DevBuf::alloc(size_t nbytes, cudaStream_t stream)
{
    release();
    s = stream;
    bytes = nbytes;
    if (nbytes == 0) nbytes = 256;
    cudaError_t e = pool_malloc(&p, nbytes, stream);
    if (e != cudaSuccess) {
        p = nullptr;
        return cuda_status(e, "cudaMallocAsync");
    }
    return TS_OK;
}

// ---------------------------------------------------------------------------------------------
// scan
// ---------------------------------------------------------------------------------------------
constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <class T>
__device__ inline T warp_incl_scan(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// Block-wide exclusive scan of one value per thread; returns the exclusive prefix, *total the sum.
template <class T, int THREADS = SCAN_THREADS>
__device__ inline T block_excl_scan(T v, T *total)
{
    __shared__ T warp_sums[THREADS / 32 + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T incl = warp_incl_scan(v);
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        T w = lane < THREADS / 32 ? warp_sums[lane] : T(0);
        T wi = warp_incl_scan(w);
        if (lane < THREADS / 32) warp_sums[lane] = wi - w;
        if (lane == THREADS / 32 - 1) warp_sums[THREADS / 32] = wi;  // total
    }
    __syncthreads();
    T excl = warp_sums[wid] + incl - v;
    if (total) *total = warp_sums[THREADS / 32];
    __syncthreads();
    return excl;
}

// Element count of a primitive: the capacity, or the smaller count held in device memory (a
// run whose size is known only on the device, e.g. a replayed CUDA graph).
__device__ __forceinline__ uint64_t dev_count(uint64_t cap, const uint32_t *n_dev)
{
    return n_dev ? min(cap, (uint64_t)*n_dev) : cap;
}

// An offset as it is stored: 64 bits as they are, 32 bits checked.
__device__ __forceinline__ void put_off(uint64_t *out, uint64_t v, uint32_t *) { *out = v; }
__device__ __forceinline__ void put_off(uint32_t *out, uint64_t v, uint32_t *status)
{
    if (v > 0xffffffffull) {
        atomicOr(status, DEV_ERR_OVERFLOW);
        v = 0xffffffffull;
    }
    *out = (uint32_t)v;
}

// Tiles of one block of a scan over n values: as many blocks as SCAN_BLOCKS at most, each with a run
// of consecutive tiles, so that a capacity far above the count costs empty blocks only up to that
// number (a plan of 33M tiles launched 16,000 blocks for 2,000 tiles) and two kernels always do.
constexpr uint64_t SCAN_BLOCKS = 152 * 8;

struct ScanPart {
    uint64_t n, first, last;  // values, tiles [first, last)
};
__device__ __forceinline__ ScanPart scan_part(uint64_t ncap, const uint32_t *n_dev)
{
    ScanPart p;
    p.n = dev_count(ncap, n_dev);
    const uint64_t tiles = p.n / SCAN_TILE + 1;  // (one of them holds index n)
    const uint64_t per = (tiles + gridDim.x - 1) / gridDim.x;
    p.first = min(tiles, per * blockIdx.x);
    p.last = min(tiles, p.first + per);
    return p;
}

__global__ void k_tile_sums(const uint32_t *in, uint64_t ncap, const uint32_t *n_dev, uint32_t mask,
                            uint64_t *sums)
{
    pdl_enter();
    const ScanPart p = scan_part(ncap, n_dev);
    uint64_t acc = 0;
    for (uint64_t t = p.first; t < p.last; t++) {
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; k++) {
            const uint64_t i = t * SCAN_TILE + (uint64_t)k * SCAN_THREADS + threadIdx.x;
            if (i < p.n) acc += in[i] & mask;
        }
    }
    uint64_t total;
    block_excl_scan<uint64_t>(acc, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// out[i] = exclusive prefix, and out[n] = total by the block whose tile holds index n. Every block
// first adds up the sums of the blocks before it.
template <class Tout>
__global__ void k_tile_scan(const uint32_t *in, uint64_t ncap, const uint32_t *n_dev, uint32_t mask,
                            const uint64_t *sums, Tout *out, uint32_t *status)
{
    pdl_enter();
    const ScanPart p = scan_part(ncap, n_dev);
    if (p.first >= p.last) return;
    uint64_t before = 0;
    if (blockIdx.x) {
        uint64_t pre = 0;
        for (uint32_t j = threadIdx.x; j < blockIdx.x; j += SCAN_THREADS) pre += sums[j];
        block_excl_scan<uint64_t>(pre, &before);
    }
    for (uint64_t t = p.first; t < p.last; t++) {
        // thread-contiguous items for a stable sequential order within a thread
        uint32_t v[SCAN_ITEMS];
        uint64_t acc = 0;
        const uint64_t tbase = t * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; k++) {
            v[k] = tbase + k < p.n ? in[tbase + k] & mask : 0u;
            acc += v[k];
        }
        uint64_t total;
        uint64_t off = before + block_excl_scan<uint64_t>(acc, &total);
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; k++) {
            if (tbase + k < p.n) put_off(out + tbase + k, off, status);
            off += v[k];
        }
        before += total;
        if (threadIdx.x == 0 && p.n < (t + 1) * SCAN_TILE) put_off(out + p.n, before, status);
    }
}

// Exclusive scan of n (or *n_dev <= n) values: out[0..n] with out[n] = total. 32-bit offsets are
// checked and written by the scan itself.
template <class Tout>
static ts_status scan_impl(const uint32_t *in, Tout *out, uint64_t n, const uint32_t *n_dev,
                           cudaStream_t s, uint32_t mask, uint32_t *status)
{
    if (n == 0) {
        TS_CUDA(cudaMemsetAsync(out, 0, sizeof(Tout), s));
        return TS_OK;
    }
    const unsigned nb = (unsigned)std::min<uint64_t>(n / SCAN_TILE + 1, SCAN_BLOCKS);
    DevBuf sums;
    if (nb > 1) {
        TS_CHECK(sums.alloc(sizeof(uint64_t) * nb, s));
        TS_LAUNCH_PDL(k_tile_sums, dim3(nb), dim3(SCAN_THREADS), 0, s,
                      in, n, n_dev, mask, sums.as<uint64_t>());
    }
    TS_LAUNCH_PDL(k_tile_scan<Tout>, dim3(nb), dim3(SCAN_THREADS), 0, s,
                  in, n, n_dev, mask, sums.as<uint64_t>(), out, status);
    return TS_OK;
}

ts_status scan_u32_to_u64(const uint32_t *in, uint64_t *out, uint64_t n, cudaStream_t s,
                          const uint32_t *n_dev, uint32_t mask)
{
    return scan_impl<uint64_t>(in, out, n, n_dev, s, mask, nullptr);
}

ts_status scan_u32(const uint32_t *in, uint32_t *out, uint64_t n, uint32_t *status,
                   cudaStream_t s, const uint32_t *n_dev)
{
    return scan_impl<uint32_t>(in, out, n, n_dev, s, ~0u, status);
}

// ---------------------------------------------------------------------------------------------
// radix sort: LSD, 8-bit digits, 1024 threads x 4 keys per block tile. Each pass: per-tile digit
// histograms, and a stable scatter in which every warp ranks its 128 consecutive keys with
// __match_any_sync and the block adds the earlier warps' counts. Up to RS_FUSED_TILES tiles (2M
// keys) the scatter adds up the histograms itself: four groups of threads, a thread per digit,
// read them tile by tile, coalesced, while the block's keys arrive. (With 2048 keys a tile and a
// thread reading a digit's counts of all tiles one after the other, that took 25 of the 31 us of
// a pass over 300,000 keys.) Above, a scan kernel turns digit-major histograms into offsets.
// Bound: L2 latency for the sizes of a search's units, HBM for an index's keys.
// ---------------------------------------------------------------------------------------------
constexpr int RS_THREADS = 1024;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ITEMS = 4;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int RS_RADIX = 256;
constexpr uint32_t RS_FUSED_TILES = 512;

template <class K, bool FUSED>
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const K *keys, uint64_t ncap,
                                                        const uint32_t *n_dev, int shift,
                                                        uint32_t *hist, uint32_t ntiles)
{
    pdl_enter();
    __shared__ uint32_t h[RS_RADIX];
    const uint64_t n = dev_count(ncap, n_dev);
    const uint64_t base = (uint64_t)blockIdx.x * RS_TILE;
    if (FUSED && base >= n) return;
    if (threadIdx.x < RS_RADIX) h[threadIdx.x] = 0;
    K key[RS_ITEMS];
#pragma unroll
    for (int k = 0; k < RS_ITEMS; k++) {
        const uint64_t i = base + (uint64_t)k * RS_THREADS + threadIdx.x;
        key[k] = i < n ? keys[i] : K(0);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RS_ITEMS; k++) {
        const uint64_t i = base + (uint64_t)k * RS_THREADS + threadIdx.x;
        const bool ok = i < n;
        const uint32_t d = (uint32_t)(key[k] >> shift) & 0xffu;
        // the lanes of a warp often share their digit (the high digits of sorted starts)
        const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
        if (__all_sync(0xffffffffu, ok && d == d0)) {
            if ((threadIdx.x & 31) == 0) atomicAdd(&h[d], 32u);
        } else if (ok) {
            atomicAdd(&h[d], 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x < RS_RADIX) {
        const uint64_t d = threadIdx.x;
        hist[FUSED ? (uint64_t)blockIdx.x * RS_RADIX + d : d * ntiles + blockIdx.x] = h[d];
    }
}

// off: the tiles' histograms (FUSED), or the scanned digit-major ones.
template <class K, bool FUSED>
__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const K *keys_in, const uint32_t *vals_in,
                                                           K *keys_out, uint32_t *vals_out,
                                                           uint64_t ncap, const uint32_t *n_dev,
                                                           int shift, const uint32_t *hist,
                                                           const uint64_t *digit_off,
                                                           uint32_t ntiles)
{
    pdl_enter();
    __shared__ uint32_t wcnt[RS_WARPS][RS_RADIX];
    __shared__ uint32_t part[2][RS_THREADS];
    __shared__ uint64_t dbase[RS_RADIX];
    const uint64_t n = dev_count(ncap, n_dev);
    if ((uint64_t)blockIdx.x * RS_TILE >= n) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t wbase = (uint64_t)blockIdx.x * RS_TILE + (uint64_t)wid * (RS_ITEMS * 32);
    K key[RS_ITEMS];
    uint32_t val[RS_ITEMS], rank[RS_ITEMS];
#pragma unroll
    for (int k = 0; k < RS_ITEMS; k++) {
        const uint64_t i = wbase + (uint64_t)k * 32 + lane;
        key[k] = i < n ? keys_in[i] : K(0);
        val[k] = i < n ? vals_in[i] : 0u;
    }
    for (int i = threadIdx.x; i < RS_WARPS * RS_RADIX; i += RS_THREADS) (&wcnt[0][0])[i] = 0;
    if (FUSED) {
        const uint32_t nt = (uint32_t)((n + RS_TILE - 1) / RS_TILE);
        const uint32_t d = threadIdx.x & (RS_RADIX - 1), grp = threadIdx.x / RS_RADIX;
        uint32_t tot = 0, pre = 0;
#pragma unroll 8
        for (uint32_t t = grp; t < nt; t += RS_THREADS / RS_RADIX) {
            const uint32_t v = hist[(uint64_t)t * RS_RADIX + d];
            tot += v;
            pre += t < blockIdx.x ? v : 0u;
        }
        part[0][threadIdx.x] = tot;
        part[1][threadIdx.x] = pre;
        __syncthreads();
        tot = pre = 0;
        if (threadIdx.x < RS_RADIX)
            for (int g = 0; g < RS_THREADS / RS_RADIX; g++) {
                tot += part[0][g * RS_RADIX + threadIdx.x];
                pre += part[1][g * RS_RADIX + threadIdx.x];
            }
        const uint32_t base = block_excl_scan<uint32_t, RS_THREADS>(tot, nullptr);
        if (threadIdx.x < RS_RADIX) dbase[threadIdx.x] = base + pre;
    } else {
        if (threadIdx.x < RS_RADIX)
            dbase[threadIdx.x] = digit_off[(uint64_t)threadIdx.x * ntiles + blockIdx.x];
        __syncthreads();
    }
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int k = 0; k < RS_ITEMS; k++) {
        const bool ok = wbase + (uint64_t)k * 32 + lane < n;
        const uint32_t dgt = ok ? ((uint32_t)(key[k] >> shift) & 0xffu) : 0x100u;
        const uint32_t peers = __match_any_sync(0xffffffffu, dgt);
        const uint32_t leader = __ffs(peers) - 1;
        uint32_t cur = 0;
        if (ok && lane == (int)leader) {
            cur = wcnt[wid][dgt];
            wcnt[wid][dgt] = cur + __popc(peers);
        }
        rank[k] = __shfl_sync(0xffffffffu, cur, leader) + __popc(peers & lt_mask);
        __syncwarp();
    }
    __syncthreads();
    // exclusive prefix over warps, per digit
    if (threadIdx.x < RS_RADIX) {
        uint32_t run = 0;
#pragma unroll 8
        for (int w = 0; w < RS_WARPS; w++) {
            const uint32_t c = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RS_ITEMS; k++) {
        if (wbase + (uint64_t)k * 32 + lane >= n) continue;
        const uint32_t dgt = (uint32_t)(key[k] >> shift) & 0xffu;
        const uint64_t dst = dbase[dgt] + wcnt[wid][dgt] + rank[k];
        keys_out[dst] = key[k];
        vals_out[dst] = val[k];
    }
}

// The whole sort of up to RS_SMALL keys in one block, pass by pass through shared memory (two
// launches and two rounds through L2 a pass cost 5 us each on a few keys).
constexpr int RS_SMALL_ITEMS = 2;
constexpr int RS_SMALL = RS_THREADS * RS_SMALL_ITEMS;

template <class K>
__global__ void __launch_bounds__(RS_THREADS) k_rs_small(K *keys, uint32_t *vals, uint64_t ncap,
                                                         const uint32_t *n_dev, int passes)
{
    pdl_enter();
    __shared__ K skey[RS_SMALL];
    __shared__ uint32_t sval[RS_SMALL];
    __shared__ uint16_t wcnt[RS_WARPS][RS_RADIX];
    __shared__ uint32_t dbase[RS_RADIX];
    const uint32_t n = (uint32_t)dev_count(ncap, n_dev);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t at = wid * (RS_SMALL_ITEMS * 32) + lane;
    const uint32_t lt_mask = (1u << lane) - 1u;
    K key[RS_SMALL_ITEMS];
    uint32_t val[RS_SMALL_ITEMS], rank[RS_SMALL_ITEMS];
#pragma unroll
    for (int k = 0; k < RS_SMALL_ITEMS; k++) {
        const uint32_t i = at + k * 32;
        key[k] = i < n ? keys[i] : K(0);
        val[k] = i < n ? vals[i] : 0u;
    }
    for (int p = 0; p < passes; p++) {
        for (int i = threadIdx.x; i < RS_WARPS * RS_RADIX / 2; i += RS_THREADS)
            reinterpret_cast<uint32_t *>(&wcnt[0][0])[i] = 0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < RS_SMALL_ITEMS; k++) {
            const bool ok = at + k * 32 < n;
            const uint32_t dgt = ok ? ((uint32_t)(key[k] >> (8 * p)) & 0xffu) : 0x100u;
            const uint32_t peers = __match_any_sync(0xffffffffu, dgt);
            const uint32_t leader = __ffs(peers) - 1;
            uint32_t cur = 0;
            if (ok && lane == (int)leader) {
                cur = wcnt[wid][dgt];
                wcnt[wid][dgt] = (uint16_t)(cur + __popc(peers));
            }
            rank[k] = __shfl_sync(0xffffffffu, cur, leader) + __popc(peers & lt_mask);
            __syncwarp();
        }
        __syncthreads();
        uint32_t run = 0;
        if (threadIdx.x < RS_RADIX) {
#pragma unroll 8
            for (int w = 0; w < RS_WARPS; w++) {
                const uint32_t c = wcnt[w][threadIdx.x];
                wcnt[w][threadIdx.x] = (uint16_t)run;
                run += c;
            }
        }
        const uint32_t base = block_excl_scan<uint32_t, RS_THREADS>(run, nullptr);
        if (threadIdx.x < RS_RADIX) dbase[threadIdx.x] = base;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < RS_SMALL_ITEMS; k++) {
            if (at + k * 32 >= n) continue;
            const uint32_t dgt = (uint32_t)(key[k] >> (8 * p)) & 0xffu;
            const uint32_t dst = dbase[dgt] + wcnt[wid][dgt] + rank[k];
            skey[dst] = key[k];
            sval[dst] = val[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < RS_SMALL_ITEMS; k++) {
            const uint32_t i = at + k * 32;
            if (i < n) {
                key[k] = skey[i];
                val[k] = sval[i];
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < RS_SMALL_ITEMS; k++) {
        const uint32_t i = at + k * 32;
        if (i < n) {
            keys[i] = key[k];
            vals[i] = val[k];
        }
    }
}

template <class K>
__global__ void k_copy_kv(const K *ks, const uint32_t *vs, K *kd, uint32_t *vd, uint64_t ncap,
                          const uint32_t *n_dev)
{
    pdl_enter();
    const uint64_t n = dev_count(ncap, n_dev);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        if (kd) kd[i] = ks[i];
        vd[i] = vs[i];
    }
}

template <class K>
static ts_status radix_sort_impl(K *keys, uint32_t *vals, uint64_t n, int bits, cudaStream_t s,
                                 const uint32_t *n_dev, bool keys_out, uint64_t vary = ~0ull)
{
    if (n <= 1 || bits <= 0) return TS_OK;
    if (n <= RS_SMALL) {
        TS_LAUNCH_PDL(k_rs_small<K>, dim3(1), dim3(RS_THREADS), 0, s, keys, vals, n, n_dev,
                      (bits + 7) / 8);
        return TS_OK;
    }
    uint32_t ntiles = (uint32_t)((n + RS_TILE - 1) / RS_TILE);
    DevBuf kb, vb, hist, off;
    TS_CHECK(kb.alloc(sizeof(K) * n, s));
    TS_CHECK(vb.alloc(sizeof(uint32_t) * n, s));
    uint64_t nh = (uint64_t)RS_RADIX * ntiles;
    TS_CHECK(hist.alloc(sizeof(uint32_t) * nh, s));
    const bool fused = ntiles <= RS_FUSED_TILES;
    if (!fused) TS_CHECK(off.alloc(sizeof(uint64_t) * (nh + 1), s));
    K *ka = keys, *kbp = kb.as<K>();
    uint32_t *va = vals, *vbp = vb.as<uint32_t>();
    // digits of the bits that vary, from the lowest of them on
    if (bits < 64) vary &= (1ull << bits) - 1;
    for (int shift = 0; shift < bits; shift += 8) {
        if (!(vary >> shift)) break;
        while (!((vary >> shift) & 1)) shift++;
        if (fused) {
            TS_LAUNCH_PDL((k_rs_hist<K, true>), dim3(ntiles), dim3(RS_THREADS), 0, s, ka, n, n_dev,
                          shift, hist.as<uint32_t>(), ntiles);
            TS_LAUNCH_PDL((k_rs_scatter<K, true>), dim3(ntiles), dim3(RS_THREADS), 0, s, ka, va,
                          kbp, vbp, n, n_dev, shift, hist.as<uint32_t>(), nullptr, ntiles);
        } else {
            TS_LAUNCH_PDL((k_rs_hist<K, false>), dim3(ntiles), dim3(RS_THREADS), 0, s, ka, n, n_dev,
                          shift, hist.as<uint32_t>(), ntiles);
            TS_CHECK(scan_u32_to_u64(hist.as<uint32_t>(), off.as<uint64_t>(), nh, s));
            TS_LAUNCH_PDL((k_rs_scatter<K, false>), dim3(ntiles), dim3(RS_THREADS), 0, s, ka, va,
                          kbp, vbp, n, n_dev, shift, nullptr, off.as<uint64_t>(), ntiles);
        }
        K *tk = ka; ka = kbp; kbp = tk;
        uint32_t *tv = va; va = vbp; vbp = tv;
    }
    if (ka != keys) {
        const unsigned cb = (unsigned)std::min<uint64_t>((n + 255) / 256, 152 * 8);
        TS_LAUNCH_PDL(k_copy_kv<K>, dim3(cb), dim3(256), 0, s, ka, va, keys_out ? keys : nullptr,
                      vals, n, n_dev);
    }
    return TS_OK;
}

ts_status radix_sort_u64(uint64_t *keys, uint32_t *vals, uint64_t n, int bits, cudaStream_t s,
                         const uint32_t *n_dev, bool keys_out, uint64_t vary)
{
    return radix_sort_impl<uint64_t>(keys, vals, n, bits, s, n_dev, keys_out, vary);
}

ts_status radix_sort_u32(uint32_t *keys, uint32_t *vals, uint64_t n, int bits, cudaStream_t s,
                         const uint32_t *n_dev, bool keys_out)
{
    return radix_sort_impl<uint32_t>(keys, vals, n, bits, s, n_dev, keys_out);
}

}  // namespace ts
