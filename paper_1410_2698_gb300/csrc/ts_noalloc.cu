// ts_noalloc.cu -- an all-pairs search that allocates no memory.
//
// Who this is for: code that runs inside a host application which owns every byte of device
// memory through its own allocator or a fixed budget (a library-side cudaMalloc would bypass that
// accounting or fail), and latency-sensitive callers for whom cudaMalloc/cudaFree, which can
// synchronise the device, are not acceptable on the request path. Such callers pass their input
// and output arrays; the only working memory is TS_NOALLOC_SCRATCH_BYTES of device memory that is
// part of this library's image (a file-scope __device__ array), which every GPU that loads the
// library holds until the process exits.
//
// Work layout: tiles of 32 query segments x 1024 database segments in the caller's order; a first
// kernel bounds every run of 32 (or more, for large databases) consecutive database segments, pass 1
// counts each tile's hits into the scratch array, a three-kernel scan turns the counts into row
// offsets (also in the scratch array), pass 2 writes the rows of the tiles that have any. The pair
// test is the same three-stage test as the indexed search (FP32 box filter, FP32 gap filter, exact
// FP64 closed form).
#include <algorithm>
#include <mutex>

#include "ts_device.cuh"

namespace ts {

namespace {

constexpr uint64_t NA_SCRATCH_BYTES = 32ull << 20;  // TS_NOALLOC_SCRATCH_BYTES
constexpr int NA_QB = 32;                           // query segments per tile
constexpr int NA_EB = 1024;                         // database segments per tile
constexpr int NA_SCAN = 2048;                       // tiles per scan block
constexpr uint64_t NA_MAX_TILES = 2500000;          // TS_NOALLOC_MAX_TILES
constexpr uint64_t NA_CTRL = 256;
constexpr uint64_t NA_COUNTS = NA_CTRL;
constexpr uint64_t NA_OFFS = (NA_COUNTS + 4 * NA_MAX_TILES + 255) / 256 * 256;
constexpr uint64_t NA_PARTS = (NA_OFFS + 8 * (NA_MAX_TILES + 1) + 255) / 256 * 256;
constexpr uint64_t NA_MAX_PARTS = (NA_MAX_TILES + NA_SCAN - 1) / NA_SCAN;
// bounding records of the runs, in what the counts and offsets leave of the scratch (106,000), and
// of the tiles' whole widths
constexpr uint64_t NA_MAX_WIDE = 4096;
constexpr uint64_t NA_WIDE = (NA_PARTS + 8 * (NA_MAX_PARTS + 1) + 255) / 256 * 256;
constexpr uint64_t NA_BOXES = NA_WIDE + NA_MAX_WIDE * sizeof(RecF);
constexpr uint64_t NA_MAX_BOXES = (NA_SCRATCH_BYTES - NA_BOXES) / sizeof(RecF);
static_assert(NA_PARTS + 8 * (NA_MAX_PARTS + 1) <= NA_SCRATCH_BYTES, "scratch layout");
static_assert(NA_MAX_PARTS <= 2048, "one block scans the partial sums");

// The scratch: shared by every call of ts_search_brute_noalloc on a device.
static __device__ __align__(256) unsigned char g_na_scratch[NA_SCRATCH_BYTES];

struct NaCtrl {
    uint32_t status;
    uint32_t pad[3];
    unsigned long long total;
};

struct NaParams {
    const double *e[8];
    const double *q[8];
    uint64_t n, nq;
    uint64_t nchunk, ntiles;
    double d, dd, Ts, Te;
    float d_up, d_dn, d2u;
    uint32_t run;            // database segments per bounding record (32 to NA_EB); 0: none kept
    uint32_t seg;            // consecutive tiles a warp takes at a time (at most 32)
    uint32_t wide;           // bounding records of the tiles' widths are kept
    uint64_t capacity;       // rows the output arrays hold (0 when one of them is missing)
    uint32_t *q_out, *e_out;
    double *tin_out, *tout_out;
    unsigned char *scratch;  // device address of g_na_scratch
};

constexpr int NA_WARPS = 4;

// What a warp keeps in shared memory: its 32 query segments, the 32 database segments it tests
// against them, and the pairs of the two that passed the FP32 filters.
struct NaWarp {
    QueryD q[NA_QB];  // filled once some pair of these queries passes the filters
    SegD e[32];
    float4 ea[NA_QB], eb[NA_QB];
    uint16_t pair[NA_QB * 32];  // member << 5 | database segment
};

__device__ __forceinline__ bool na_valid(const double v[8])
{
    bool fin = true;
    for (int k = 0; k < 8; k++) fin = fin && isfinite(v[k]);
    return fin && v[7] > v[3];
}

__device__ __forceinline__ RecF na_rec(const double v[8])
{
    RecF r;
    r.xmin = __double2float_rd(fmin(v[0], v[4])); r.xmax = __double2float_ru(fmax(v[0], v[4]));
    r.ymin = __double2float_rd(fmin(v[1], v[5])); r.ymax = __double2float_ru(fmax(v[1], v[5]));
    r.zmin = __double2float_rd(fmin(v[2], v[6])); r.zmax = __double2float_ru(fmax(v[2], v[6]));
    r.t0 = __double2float_rd(v[3]);
    r.t1 = __double2float_ru(v[7]);
    return r;
}

// lo = minimum of lo over the warp's lanes, hi = maximum (four components each)
__device__ __forceinline__ void na_warp_bounds(float lo[4], float hi[4])
{
#pragma unroll
    for (int o = 16; o; o >>= 1)
#pragma unroll
        for (int k = 0; k < 4; k++) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
}

// Validation of the database and the bounding record of every run of P.run consecutive segments
// (segments of one trajectory are usually neighbours, so a run is short in time and space). A warp
// per run. Bound: HBM, 64 B read per segment, once per call.
__global__ void __launch_bounds__(256) k_na_boxes(NaParams P)
{
    NaCtrl *ctrl = reinterpret_cast<NaCtrl *>(P.scratch);
    RecF *box = reinterpret_cast<RecF *>(P.scratch + NA_BOXES);
    const int lane = threadIdx.x & 31;
    const uint64_t step = P.run ? P.run : 32;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t c = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c * step < P.n;
         c += warps) {
        float lo[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
        float hi[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        for (uint64_t i = c * step + lane; i < (c + 1) * step && i < P.n; i += 32) {
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; k++) v[k] = P.e[k][i];
            if (!na_valid(v)) {  // (the call ends with an error: its boxes do not matter)
                atomicOr(&ctrl->status, DEV_ERR_INVALID);
                continue;
            }
            const RecF r = na_rec(v);
            lo[0] = fminf(lo[0], r.xmin); hi[0] = fmaxf(hi[0], r.xmax);
            lo[1] = fminf(lo[1], r.ymin); hi[1] = fmaxf(hi[1], r.ymax);
            lo[2] = fminf(lo[2], r.zmin); hi[2] = fmaxf(hi[2], r.zmax);
            lo[3] = fminf(lo[3], r.t0); hi[3] = fmaxf(hi[3], r.t1);
        }
        if (!P.run) continue;
        na_warp_bounds(lo, hi);
        if (lane == 0) {
            RecF b;
            b.xmin = lo[0]; b.xmax = hi[0];
            b.ymin = lo[1]; b.ymax = hi[1];
            b.zmin = lo[2]; b.zmax = hi[2];
            b.t0 = lo[3]; b.t1 = hi[3];
            box[c] = b;
        }
    }
}

// Bounding record of every 1024 consecutive segments, from those of their runs, a warp per record.
__global__ void __launch_bounds__(256) k_na_wide(NaParams P)
{
    const float4 *box = reinterpret_cast<const float4 *>(P.scratch + NA_BOXES);
    RecF *wide = reinterpret_cast<RecF *>(P.scratch + NA_WIDE);
    const int lane = threadIdx.x & 31;
    const uint64_t ch = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (ch >= P.nchunk) return;
    // (the lanes past the last segment repeat the last run's)
    const uint64_t i = min(ch * NA_EB + (uint64_t)lane * 32, P.n - 1);
    const float4 u = box[2 * (i / P.run)], w = box[2 * (i / P.run) + 1];
    float lo[4] = {u.x, u.z, w.x, w.z}, hi[4] = {u.y, u.w, w.y, w.w};
    na_warp_bounds(lo, hi);
    if (lane == 0) {
        RecF b;
        b.xmin = lo[0]; b.xmax = hi[0];
        b.ymin = lo[1]; b.ymax = hi[1];
        b.zmin = lo[2]; b.zmax = hi[2];
        b.t0 = lo[3]; b.t1 = hi[3];
        wide[ch] = b;
    }
}

// A warp takes P.seg consecutive tiles of one block of 32 query segments, which are prepared once,
// one per lane. First a lane per tile: does its whole width meet the bounds of the queries (pass 0),
// has it rows (pass 1)? A tile that passes is 32 blocks of 32 database segments: every lane tests
// one block's bounding record against the bounds of all 32 queries, then the blocks that pass are
// tested against each query, and only a block that some query meets is read (a lane per segment)
// and filtered, member by member; the survivors are listed in (member, lane) order and go through
// the exact test 32 at a time. Rows of a tile are in (block, member, lane) order.
//
// Bound: latency and issue on sparse data (a tile that no query meets costs a lane one load and one
// test), the FP32 filters where every block is met. The two passes on 10,000 x 200,000 segments of
// random walks took 6.51 + 7.73 ms when every tile converted and tested all its segments and
// prepared its queries, 0.083 + 0.031 ms when a warp looked at every tile, 0.066 + 0.028 ms now.
template <int PASS>
__global__ void __launch_bounds__(NA_WARPS * 32) k_na_tiles(NaParams P)
{
    __shared__ NaWarp smem[NA_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    NaWarp &W = smem[wid];
    const unsigned FULL = 0xffffffffu;
    const uint32_t lt_mask = (1u << lane) - 1u;
    NaCtrl *ctrl = reinterpret_cast<NaCtrl *>(P.scratch);
    uint32_t *counts = reinterpret_cast<uint32_t *>(P.scratch + NA_COUNTS);
    const unsigned long long *offs = reinterpret_cast<const unsigned long long *>(P.scratch + NA_OFFS);
    const float4 *box = reinterpret_cast<const float4 *>(P.scratch + NA_BOXES);
    const float4 *wide = reinterpret_cast<const float4 *>(P.scratch + NA_WIDE);
    const uint64_t nwin = (P.nchunk + P.seg - 1) / P.seg;
    const uint64_t units = P.ntiles / P.nchunk * nwin;
    uint64_t qb = ~0ull;              // query block in the lanes
    bool live = false, have_q = false;
    float4 ea = make_float4(0.f, 0.f, 0.f, 0.f), eb = ea, ga = ea, gb = ea;
    if (PASS == 1 && (ctrl->total > P.capacity || ctrl->status)) return;  // (no rows)
    for (uint64_t u = (uint64_t)blockIdx.x * NA_WARPS + wid; u < units;
         u += (uint64_t)gridDim.x * NA_WARPS) {
        // a lane per tile
        const uint64_t ch0 = u % nwin * P.seg, tl = u / nwin * P.nchunk + ch0 + lane;
        const bool in = (uint32_t)lane < P.seg && ch0 + lane < P.nchunk;
        unsigned long long wb = 0, we = 0;
        if (PASS == 1) {
            if (in) {
                wb = offs[tl];
                we = offs[tl + 1];
            }
            if (!__ballot_sync(FULL, wb != we)) continue;
        }
        const uint64_t qi = u / nwin * NA_QB + lane;
        if (u / nwin != qb) {  // the next 32 query segments, one per lane
            qb = u / nwin;
            have_q = live = false;
            if (qi < P.nq) {
                double v[8];
#pragma unroll
                for (int k = 0; k < 8; k++) v[k] = P.q[k][qi];
                const bool ok = na_valid(v);
                if (!ok) atomicOr(&ctrl->status, DEV_ERR_INVALID);
                const RecF r = na_rec(v);
                const double w0 = dmx(v[3], P.Ts), w1 = dmn(v[7], P.Te);
                ea = make_float4(__fsub_rd(r.xmin, P.d_up), __fsub_rd(r.ymin, P.d_up),
                                 __fsub_rd(r.zmin, P.d_up), __double2float_rd(w0));
                eb = make_float4(__fadd_ru(r.xmax, P.d_up), __fadd_ru(r.ymax, P.d_up),
                                 __fadd_ru(r.zmax, P.d_up), __double2float_ru(w1));
                live = ok && w0 < w1;
            }
            W.ea[lane] = ea;
            W.eb[lane] = eb;
            float lo[4] = {live ? ea.x : INFINITY, live ? ea.y : INFINITY, live ? ea.z : INFINITY,
                           live ? ea.w : INFINITY};
            float hi[4] = {live ? eb.x : -INFINITY, live ? eb.y : -INFINITY,
                           live ? eb.z : -INFINITY, live ? eb.w : -INFINITY};
            na_warp_bounds(lo, hi);
            ga = make_float4(lo[0], lo[1], lo[2], lo[3]);
            gb = make_float4(hi[0], hi[1], hi[2], hi[3]);
            __syncwarp();
        }
        bool meet = PASS == 1 ? wb != we : in;
        if (PASS == 0 && in) {
            if (P.wide) {
                const float4 x = wide[2 * (ch0 + lane)], y = wide[2 * (ch0 + lane) + 1];
                RecF b;
                b.xmin = x.x; b.xmax = x.y; b.ymin = x.z; b.ymax = x.w;
                b.zmin = y.x; b.zmax = y.y; b.t0 = y.z; b.t1 = y.w;
                meet = filter_box(b, ga, gb);
            }
            if (!meet) counts[tl] = 0;
        }
        for (unsigned tiles = __ballot_sync(FULL, meet); tiles; tiles &= tiles - 1u) {
            const int l = __ffs(tiles) - 1;
            const uint64_t t = __shfl_sync(FULL, (unsigned long long)tl, l), e0 = (ch0 + l) * NA_EB;
            const unsigned long long wbase = __shfl_sync(FULL, wb, l), wend = __shfl_sync(FULL, we, l);
            // blocks of the tile that meet the bounds of the queries, a lane per block
            const uint32_t nent = (uint32_t)((P.n - e0) < NA_EB ? (P.n - e0) : NA_EB);
            const bool inblk = (uint32_t)lane * 32 < nent;
            RecF bx;
            bx.xmin = bx.ymin = bx.zmin = bx.t0 = -INFINITY;
            bx.xmax = bx.ymax = bx.zmax = bx.t1 = INFINITY;
            if (P.run && inblk) {
                const uint64_t c = (e0 + (uint32_t)lane * 32) / P.run;
                const float4 u = box[2 * c], w = box[2 * c + 1];
                bx.xmin = u.x; bx.xmax = u.y; bx.ymin = u.z; bx.ymax = u.w;
                bx.zmin = w.x; bx.zmax = w.y; bx.t0 = w.z; bx.t1 = w.w;
            }
            unsigned todo = __ballot_sync(FULL, inblk && filter_box(bx, ga, gb));
            unsigned long long hits = 0;
            for (; todo; todo &= todo - 1u) {
                const int c = __ffs(todo) - 1;
                RecF cb;  // block c's record, for every lane's own query
                cb.xmin = __shfl_sync(FULL, bx.xmin, c); cb.xmax = __shfl_sync(FULL, bx.xmax, c);
                cb.ymin = __shfl_sync(FULL, bx.ymin, c); cb.ymax = __shfl_sync(FULL, bx.ymax, c);
                cb.zmin = __shfl_sync(FULL, bx.zmin, c); cb.zmax = __shfl_sync(FULL, bx.zmax, c);
                cb.t0 = __shfl_sync(FULL, bx.t0, c); cb.t1 = __shfl_sync(FULL, bx.t1, c);
                unsigned act = __ballot_sync(FULL, live && filter_box(cb, ea, eb));
                if (!act) continue;
                const uint32_t j = (uint32_t)c * 32 + lane;
                const bool inb = j < nent;
                const uint64_t ei = e0 + (inb ? j : 0);
                double v[8];
#pragma unroll
                for (int k = 0; k < 8; k++) v[k] = P.e[k][ei];
                const bool use = inb && na_valid(v);
                const RecF r = na_rec(v);
                uint32_t np = 0;  // listed pairs (warp-uniform)
                for (; act; act &= act - 1u) {
                    const int m = __ffs(act) - 1;
                    const float4 mea = W.ea[m], meb = W.eb[m];
                    const bool p = use && filter_box(r, mea, meb) &&
                                   filter_gap_e(r, mea, meb, P.d_dn, P.d2u);
                    const unsigned pm = __ballot_sync(FULL, p);
                    if (p) W.pair[np + __popc(pm & lt_mask)] = (uint16_t)(m << 5 | lane);
                    np += __popc(pm);
                }
                if (!np) continue;
                {
                    const double dt = v[7] - v[3];
                    SegD e;
                    e.x0 = v[0]; e.y0 = v[1]; e.z0 = v[2]; e.t0 = v[3]; e.t1 = v[7];
                    e.vx = (v[4] - v[0]) / dt;
                    e.vy = (v[5] - v[1]) / dt;
                    e.vz = (v[6] - v[2]) / dt;
                    W.e[lane] = e;
                }
                if (!have_q) {
                    have_q = true;
                    if (qi < P.nq) {
#pragma unroll
                        for (int k = 0; k < 8; k++) v[k] = P.q[k][qi];
                        const double dt = v[7] - v[3];
                        QueryD q;
                        q.vx = (v[4] - v[0]) / dt;
                        q.vy = (v[5] - v[1]) / dt;
                        q.vz = (v[6] - v[2]) / dt;
                        q.w0 = dmx(v[3], P.Ts);
                        q.w1 = dmn(v[7], P.Te);
                        const double dw = q.w0 - v[3];  // 0 unless the interval clips the start
                        q.xw = fma(q.vx, dw, v[0]);
                        q.yw = fma(q.vy, dw, v[1]);
                        q.zw = fma(q.vz, dw, v[2]);
                        q.ndd = -P.dd;
                        W.q[lane] = q;
                    }
                }
                __syncwarp();
                for (uint32_t b = 0; b < np; b += 32) {
                    bool h = false;
                    double tin = 0.0, tout = 0.0;
                    uint32_t pr = 0;
                    if (b + lane < np) {
                        pr = W.pair[b + lane];
                        h = pair_test(W.q[pr >> 5], W.e[pr & 31u], PASS == 1, &tin, &tout);
                    }
                    const unsigned hm = __ballot_sync(FULL, h);
                    if (PASS == 1 && h) {
                        const unsigned long long o = wbase + hits + __popc(hm & lt_mask);
                        if (o < wend) {
                            P.q_out[o] = (uint32_t)(qb * NA_QB + (pr >> 5));
                            P.e_out[o] = (uint32_t)(e0 + (uint32_t)c * 32 + (pr & 31u));
                            P.tin_out[o] = tin;
                            P.tout_out[o] = tout;
                        }
                    }
                    hits += __popc(hm);
                }
                __syncwarp();
            }
            if (PASS == 0) {
                if (lane == 0) counts[t] = (uint32_t)hits;  // (at most 32 x 1024)
            } else {
                if (lane == 0 && wbase + hits != wend) atomicOr(&ctrl->status, DEV_ERR_INTERNAL);
            }
            __syncwarp();
        }
    }
}

// Scan of the tile counts into row offsets, in three launches that use only the scratch array.
__device__ __forceinline__ unsigned long long na_block_scan(unsigned long long v,
                                                            unsigned long long *total)
{
    __shared__ unsigned long long ws[33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long w = lane < nw ? ws[lane] : 0ull;
        unsigned long long wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < nw) ws[lane] = wi - w;
        if (lane == 31) ws[32] = wi;
    }
    __syncthreads();
    const unsigned long long r = ws[wid] + x - v;
    *total = ws[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(1024) k_na_scan_parts(unsigned char *scratch, uint64_t ntiles)
{
    const uint32_t *counts = reinterpret_cast<const uint32_t *>(scratch + NA_COUNTS);
    unsigned long long *parts = reinterpret_cast<unsigned long long *>(scratch + NA_PARTS);
    unsigned long long s = 0;
    const uint64_t base = (uint64_t)blockIdx.x * NA_SCAN;
    for (uint64_t k = threadIdx.x; k < NA_SCAN; k += blockDim.x)
        if (base + k < ntiles) s += counts[base + k];
    unsigned long long tot;
    na_block_scan(s, &tot);
    if (threadIdx.x == 0) parts[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_na_scan_top(unsigned char *scratch, uint64_t nparts)
{
    unsigned long long *parts = reinterpret_cast<unsigned long long *>(scratch + NA_PARTS);
    NaCtrl *ctrl = reinterpret_cast<NaCtrl *>(scratch);
    // two parts per thread, in order
    const uint64_t a = 2 * threadIdx.x, b = a + 1;
    const unsigned long long va = a < nparts ? parts[a] : 0ull, vb = b < nparts ? parts[b] : 0ull;
    unsigned long long tot;
    const unsigned long long ex = na_block_scan(va + vb, &tot);
    if (a < nparts) parts[a] = ex;
    if (b < nparts) parts[b] = ex + va;
    if (threadIdx.x == 0) ctrl->total = tot;
}

__global__ void __launch_bounds__(1024) k_na_scan_final(unsigned char *scratch, uint64_t ntiles)
{
    const uint32_t *counts = reinterpret_cast<const uint32_t *>(scratch + NA_COUNTS);
    unsigned long long *offs = reinterpret_cast<unsigned long long *>(scratch + NA_OFFS);
    const unsigned long long *parts = reinterpret_cast<const unsigned long long *>(scratch + NA_PARTS);
    const NaCtrl *ctrl = reinterpret_cast<const NaCtrl *>(scratch);
    const uint64_t base = (uint64_t)blockIdx.x * NA_SCAN;
    // two consecutive tiles per thread
    const uint64_t a = base + 2 * threadIdx.x, b = a + 1;
    const unsigned long long va = a < ntiles ? counts[a] : 0ull, vb = b < ntiles ? counts[b] : 0ull;
    unsigned long long tot;
    const unsigned long long ex = parts[blockIdx.x] + na_block_scan(va + vb, &tot);
    if (a < ntiles) offs[a] = ex;
    if (b < ntiles) offs[b] = ex + va;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) offs[ntiles] = ctrl->total;
}

// Device address of g_na_scratch per device, looked up once per device (with that device
// current) on the first call that runs on it.
std::mutex g_na_mu;
unsigned char *g_na_ptr[256] = {nullptr};

ts_status na_scratch(unsigned char **out)
{
    int dev = 0;
    TS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) {
        set_error("ts_search_brute_noalloc: device ordinal %d out of range", dev);
        return TS_ERR_INVALID_ARG;
    }
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_na_scratch);
        if (e != cudaSuccess || !p) return cuda_status(e, "cudaGetSymbolAddress(g_na_scratch)");
        g_na_ptr[dev] = static_cast<unsigned char *>(p);
    }
    *out = g_na_ptr[dev];
    return TS_OK;
}

float na_float_up(double x)
{
    float f = (float)x;
    if ((double)f < x) f = nextafterf(f, INFINITY);
    return f;
}

float na_float_dn(double x)
{
    float f = (float)x;
    if ((double)f > x) f = nextafterf(f, -INFINITY);
    return f;
}

ts_status na_status(uint32_t st)
{
    if (st & DEV_ERR_INVALID) {
        set_error("invalid segment (NaN/Inf or t_end <= t_start)");
        return TS_ERR_INVALID_ARG;
    }
    if (st & DEV_ERR_OVERFLOW) {
        set_error("a tile's hit count does not fit in 32 bits");
        return TS_ERR_CAPACITY;
    }
    if (st) {
        set_error("no-allocation search: device status 0x%x", st);
        return TS_ERR_INTERNAL;
    }
    return TS_OK;
}

}  // namespace

ts_status search_brute_noalloc(const ts_segments *db, const ts_segments *q,
                               const ts_query_params *qp, uint32_t *q_idx, uint32_t *e_idx,
                               double *t_in, double *t_out, uint64_t capacity, uint64_t *count,
                               cudaStream_t s)
{
    if (!db || !q || !qp || !count) {
        set_error("ts_search_brute_noalloc: NULL argument");
        return TS_ERR_INVALID_ARG;
    }
    *count = 0;
    if (db->on_host || q->on_host) {
        set_error("ts_search_brute_noalloc: inputs must be device pointers (on_host = 0)");
        return TS_ERR_INVALID_ARG;
    }
    if (!(qp->d > 0.0) || !isfinite(qp->d) || isnan(qp->t_start) || isnan(qp->t_end) ||
        qp->t_start > qp->t_end) {
        set_error("ts_search_brute_noalloc: need finite d > 0 and t_start <= t_end");
        return TS_ERR_INVALID_ARG;
    }
    if (db->n > 0xffffffffull || q->n > 0xffffffffull) {
        set_error("ts_search_brute_noalloc: sizes above 2^32 - 1");
        return TS_ERR_INVALID_ARG;
    }
    const double *ec[8] = {db->x0, db->y0, db->z0, db->t0, db->x1, db->y1, db->z1, db->t1};
    const double *qc[8] = {q->x0, q->y0, q->z0, q->t0, q->x1, q->y1, q->z1, q->t1};
    for (int k = 0; k < 8; k++)
        if ((db->n && !ec[k]) || (q->n && !qc[k])) {
            set_error("ts_search_brute_noalloc: NULL column %d", k);
            return TS_ERR_INVALID_ARG;
        }
    if (db->n == 0 || q->n == 0) return TS_OK;
    const uint64_t nchunk = (db->n + NA_EB - 1) / NA_EB;
    const uint64_t ntiles = (q->n + NA_QB - 1) / NA_QB * nchunk;
    if (ntiles > NA_MAX_TILES) {
        set_error("ts_search_brute_noalloc: %llu tiles of 32 query x 1024 database segments "
                  "exceed the fixed scratch limit of %llu tiles",
                  (unsigned long long)ntiles, (unsigned long long)NA_MAX_TILES);
        return TS_ERR_CAPACITY;
    }
    unsigned char *scratch = nullptr;
    TS_CHECK(na_scratch(&scratch));
    NaParams P;
    for (int k = 0; k < 8; k++) {
        P.e[k] = ec[k];
        P.q[k] = qc[k];
    }
    P.n = db->n;
    P.nq = q->n;
    P.nchunk = nchunk;
    P.ntiles = ntiles;
    P.d = qp->d;
    P.dd = qp->d * qp->d;
    P.Ts = qp->t_start;
    P.Te = qp->t_end;
    P.d_up = na_float_up(qp->d);
    P.d_dn = na_float_dn(qp->d);
    P.d2u = na_float_up(P.dd * (1.0 + 1e-6));
    // the finest runs whose bounding records fit; none above NA_MAX_BOXES tiles' width
    P.run = 32;
    while (P.run < (uint32_t)NA_EB && (db->n + P.run - 1) / P.run > NA_MAX_BOXES) P.run *= 2;
    if ((db->n + P.run - 1) / P.run > NA_MAX_BOXES) P.run = 0;
    P.q_out = q_idx;
    P.e_out = e_idx;
    P.tin_out = t_in;
    P.tout_out = t_out;
    P.scratch = scratch;
    int dev = 0, sms = 0;
    TS_CUDA(cudaGetDevice(&dev));
    TS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const uint64_t want = (ntiles + NA_WARPS - 1) / NA_WARPS;
    const unsigned grid = (unsigned)(want < (uint64_t)sms * 6 ? want : (uint64_t)sms * 6);
    // consecutive tiles per warp: as many as leave every warp a turn
    const uint64_t seg = ntiles / ((uint64_t)grid * NA_WARPS);
    P.seg = (uint32_t)(seg < 1 ? 1 : (seg > 32 ? 32 : seg));
    P.wide = P.run && nchunk <= NA_MAX_WIDE;
    const bool out_ok = q_idx && e_idx && t_in && t_out;
    P.capacity = out_ok ? capacity : 0;
    const uint64_t runs = (db->n + 31) / 32;
    const unsigned bgrid = (unsigned)std::min<uint64_t>((runs + 7) / 8, (uint64_t)sms * 16);
    const uint64_t nparts = (ntiles + NA_SCAN - 1) / NA_SCAN;

    // the control words start at zero on every call; counts and offsets are fully rewritten
    TS_CUDA(cudaMemsetAsync(scratch, 0, NA_CTRL, s));
    k_na_boxes<<<bgrid, 256, 0, s>>>(P);
    TS_LAUNCHED();
    if (P.wide) {
        k_na_wide<<<(unsigned)((nchunk + 7) / 8), 256, 0, s>>>(P);
        TS_LAUNCHED();
    }
    k_na_tiles<0><<<grid, NA_WARPS * 32, 0, s>>>(P);
    TS_LAUNCHED();
    k_na_scan_parts<<<(unsigned)nparts, 1024, 0, s>>>(scratch, ntiles);
    TS_LAUNCHED();
    k_na_scan_top<<<1, 1024, 0, s>>>(scratch, nparts);
    TS_LAUNCHED();
    k_na_scan_final<<<(unsigned)nparts, 1024, 0, s>>>(scratch, ntiles);
    TS_LAUNCHED();
    // (the device sees whether the rows fit: one wait, for the outcome of both passes)
    k_na_tiles<1><<<grid, NA_WARPS * 32, 0, s>>>(P);
    TS_LAUNCHED();
    NaCtrl h;
    TS_CUDA(cudaMemcpyAsync(&h, scratch, sizeof(NaCtrl), cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    TS_CHECK(na_status(h.status));
    *count = h.total;
    if (h.total > capacity) {
        set_error("ts_search_brute_noalloc: %llu result rows exceed the capacity %llu",
                  (unsigned long long)h.total, (unsigned long long)capacity);
        return TS_ERR_CAPACITY;
    }
    if (h.total && !out_ok) {
        set_error("ts_search_brute_noalloc: NULL output array");
        return TS_ERR_INVALID_ARG;
    }
    return TS_OK;
}

}  // namespace ts
