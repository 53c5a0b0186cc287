// ts_index.cu -- building the resident index on the device.
//
// Steps (all device kernels; the host only picks parameters from exact reductions):
//   ingest   : validate (finite, t1 > t0), order keys of t_start, exact extents   (Sec. 3.1)
//   sort     : stable radix sort by t_start, ties by input index                     (Sec. 4.2)
//   parts    : temporal bin and subbins or cell of every entry, in the input's order
//   gather   : FP64 exact records (velocity precomputed) and FP32 outward-rounded
//              prefilter records in sorted order
//   bins     : m temporal bins, B_j^start, B_j^end, first/last offsets, prefix max   (Sec. 4.2)
//   subbins  : per dimension, (subbin, entry) keys -> radix sort -> X/Y/Z id arrays and
//              (subbin, bin) offsets                                                 (Sec. 4.3)
//   grid     : per entry its MBB's cells -> (cell, entry) keys -> radix sort -> lookup array A
//              and dense cell offsets                                                (Sec. 4.1)
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ts_index.cuh"

namespace ts {

namespace {

constexpr int TPB = 256;

inline unsigned nblocks(uint64_t n, int tpb = TPB)
{
    uint64_t b = (n + tpb - 1) / tpb;
    return (unsigned)(b ? b : 1);
}

// reduction slots (order keys): 0 min t0, 1 max t1, 2 max duration, 3..5 min emin, 6..8 max
// emax, 9..11 max extent
// 12 the bits in which some t0's key differs from the first's
enum { R_TMIN = 0, R_TMAX = 1, R_DUR = 2, R_EMIN = 3, R_EMAX = 6, R_LONG = 9, R_VARY = 12, R_N = 13 };

// (on the integer pipe)
__device__ inline bool finite_d(double x)
{
    return ((uint32_t)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}

__device__ inline unsigned long long warp_max_u64(unsigned long long v)
{
    for (int o = 16; o; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}

struct SegIn {
    const double *f[8];
};

__global__ void k_init_red(unsigned long long *red)
{
    int i = threadIdx.x;
    if (i >= R_N) return;
    bool is_min = (i == R_TMIN) || (i >= R_EMIN && i < R_EMIN + 3);
    red[i] = is_min ? ~0ull : 0ull;
}

// Grid-stride, the extremes in registers and one atomic per block and extreme: an atomic per warp
// and extreme on these 12 addresses took 230 of 244 us for 1M segments. Comparisons are made on
// the order keys, integers; four FP64 subtractions are left. Bound: HBM (64 B read, 12 written).
__global__ void __launch_bounds__(TPB) k_ingest(SegIn in, uint64_t n, uint64_t *keys, uint32_t *vals,
                                                unsigned long long *red, uint32_t *status)
{
    unsigned long long r[R_N];
#pragma unroll
    for (int k = 0; k < R_N; k++) r[k] = (k == R_TMIN || (k >= R_EMIN && k < R_EMIN + 3)) ? ~0ull : 0ull;
    const uint64_t first = dkey(in.f[3][0]);
    bool bad = false;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = in.f[k][i];
        bool valid = true;
        unsigned long long key[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            valid = valid && finite_d(v[k]);
            key[k] = dkey(v[k]);
        }
        valid = valid && key[7] > key[3];
        bad = bad || !valid;
        keys[i] = key[3];
        vals[i] = (uint32_t)i;
        r[R_VARY] |= key[3] ^ first;
        if (!valid) continue;
        r[R_TMIN] = min(r[R_TMIN], key[3]);
        r[R_TMAX] = max(r[R_TMAX], key[7]);
        r[R_DUR] = max(r[R_DUR], (unsigned long long)dkey(v[7] - v[3]));
#pragma unroll
        for (int d = 0; d < 3; d++) {
            r[R_EMIN + d] = min(r[R_EMIN + d], min(key[d], key[4 + d]));
            r[R_EMAX + d] = max(r[R_EMAX + d], max(key[d], key[4 + d]));
            r[R_LONG + d] = max(r[R_LONG + d], (unsigned long long)dkey(fabs(v[4 + d] - v[d])));
        }
    }
    if (bad) atomicOr(status, DEV_ERR_INVALID);
    __shared__ unsigned long long part[R_N][TPB / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < R_N; k++) {
        const bool is_min = k == R_TMIN || (k >= R_EMIN && k < R_EMIN + 3);
        unsigned long long w = r[k];
        for (int o = 16; o; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, w, o);
            w = k == R_VARY ? (w | x) : (is_min ? min(w, x) : max(w, x));
        }
        if (lane == 0) part[k][wid] = w;
    }
    __syncthreads();
    if (threadIdx.x < R_N) {
        const int k = threadIdx.x;
        const bool is_min = k == R_TMIN || (k >= R_EMIN && k < R_EMIN + 3);
        unsigned long long w = part[k][0];
        for (int j = 1; j < TPB / 32; j++) {
            const unsigned long long x = part[k][j];
            w = k == R_VARY ? (w | x) : (is_min ? min(w, x) : max(w, x));
        }
        if (k == R_VARY) atomicOr(&red[k], w);
        else if (is_min) atomicMin(&red[k], w);
        else atomicMax(&red[k], w);
    }
}

// A 1-D partition on the device: part_of from its boundary table (lo + j*w, j = 0..v).
struct PartTab {
    const double *bd;
    double lo, w;
    float iw;  // ~ 1/w, for the first guess; 0 where it has no FP32 value: part_of itself
    int v;

    // The same part as part_of: a guess in FP32 corrected by comparisons with the boundaries, made
    // on the order keys (a division and the comparisons in FP64 took 90 us for a dimension of 1M
    // entries, ten times what reading them takes).
    __device__ __forceinline__ int of(double x) const
    {
        if (v <= 1 || iw == 0.0f) return part_of(x, lo, w, v);
        const uint64_t kx = dkey(x);
        if (kx < dkey(bd[0])) return -1;
        const float f = floorf(((float)(x - lo)) * iw);
        int j = !(f < (float)v) ? v - 1 : (f < 0.0f ? 0 : (int)f);
        while (j + 1 < v && dkey(bd[j + 1]) <= kx) j++;
        while (j > 0 && dkey(bd[j]) > kx) j--;
        return j;
    }
};

__global__ void k_bounds(double *bd, double lo, double w, uint32_t v)
{
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j <= v) bd[j] = part_bound(lo, w, (int)j);
}

// Temporal bin, and the parts of the MBB's corners in the three axes: first | last << 16 (subbins),
// or the cell of the minimum corner (grid), of every entry in the input's order.
__global__ void k_parts(SegIn in, uint64_t n, PartTab bins, PartTab px, PartTab py, PartTab pz,
                        int kind, uint32_t *bin_in, uint32_t *part_in)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int j = bins.of(in.f[3][i]);
    bin_in[i] = (uint32_t)(j < 0 ? 0 : j);  // (t0 >= tmin always)
    if (kind != TS_INDEX_SPATIOTEMPORAL && kind != TS_INDEX_SPATIAL) return;
    uint32_t cell = 0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const PartTab &p = d == 0 ? px : (d == 1 ? py : pz);
        const int a = p.of(in.f[d][i]), b = p.of(in.f[4 + d][i]);
        const int lo = max(min(a, b), 0), hi = max(a, b);
        if (kind == TS_INDEX_SPATIAL) cell = cell * (uint32_t)p.v + (uint32_t)lo;
        else part_in[(uint64_t)d * n + i] = (uint32_t)lo | ((uint32_t)max(hi, 0) << 16);
    }
    if (kind == TS_INDEX_SPATIAL) part_in[i] = cell;
}

// Outward rounding of an FP64 interval to FP32 (conservative prefilter boxes).
__device__ inline float f_dn(double x) { return __double2float_rd(x); }
__device__ inline float f_up(double x) { return __double2float_ru(x); }

__global__ void k_gather(SegIn in, uint64_t n, const uint32_t *perm, const uint32_t *bin_in,
                         SegD *seg, RecF *rec, uint32_t *orig, uint32_t *bin_of,
                         unsigned long long *end_key)
{
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = s < n;
    const uint32_t i = perm[on ? s : n - 1];
    double x0 = in.f[0][i], y0 = in.f[1][i], z0 = in.f[2][i], t0 = in.f[3][i];
    double x1 = in.f[4][i], y1 = in.f[5][i], z1 = in.f[6][i], t1 = in.f[7][i];
    double dt = t1 - t0;
    SegD d;
    d.x0 = x0; d.y0 = y0; d.z0 = z0; d.t0 = t0; d.t1 = t1;
    d.vx = (x1 - x0) / dt;
    d.vy = (y1 - y0) / dt;
    d.vz = (z1 - z0) / dt;
    RecF r;
    r.xmin = f_dn(fmin(x0, x1)); r.xmax = f_up(fmax(x0, x1));
    r.ymin = f_dn(fmin(y0, y1)); r.ymax = f_up(fmax(y0, y1));
    r.zmin = f_dn(fmin(z0, z1)); r.zmax = f_up(fmax(z0, z1));
    r.t0 = f_dn(t0); r.t1 = f_up(t1);
    const uint32_t j = bin_in[i];
    if (on) {
        seg[s] = d;
        rec[s] = r;
        orig[s] = i;
        bin_of[s] = j;
    }
    // the bin's latest end: one atomic for a warp of one bin (the lanes are in start order)
    const unsigned FULL = 0xffffffffu;
    const unsigned long long k = dkey(t1);
    if (__all_sync(FULL, j == __shfl_sync(FULL, j, 0))) {
        const unsigned long long w = warp_max_u64(k);
        if ((threadIdx.x & 31) == 0) atomicMax(&end_key[j], w);
    } else {
        atomicMax(&end_key[j], k);
    }
}

// Key of an entry inside its bin: (bin, Morton code of its FP32 box centre, `bits` per axis). Any
// order inside a bin leaves every bin's range unchanged; along the Morton curve 64 consecutive
// entries are near each other in all three axes, so a chunk's bounding record rejects most
// queries (ordered by x alone, a chunk was a slab of the whole y-z extent).
__global__ void k_tm_key(const RecF *rec, const uint32_t *bin_of, uint64_t n, MortonMap mm,
                         uint64_t *keys, uint32_t *vals)
{
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const RecF r = rec[s];
    keys[s] = ((uint64_t)bin_of[s] << (3 * mm.bits)) |
              mm.code(0.5f * r.xmin + 0.5f * r.xmax, 0.5f * r.ymin + 0.5f * r.ymax,
                      0.5f * r.zmin + 0.5f * r.zmax);
    vals[s] = (uint32_t)s;
}

// Entries (every stride-th) by their place along each axis.
__global__ void __launch_bounds__(TPB) k_axis_hist(const RecF *rec, uint64_t n, uint64_t stride,
                                                   MortonMap mm, uint32_t *hist)
{
    __shared__ uint32_t h[3 * AXIS_BINS];
    for (int i = threadIdx.x; i < 3 * AXIS_BINS; i += TPB) h[i] = 0;
    __syncthreads();
    for (uint64_t i = ((uint64_t)blockIdx.x * TPB + threadIdx.x) * stride; i < n;
         i += (uint64_t)gridDim.x * TPB * stride) {
        const RecF r = rec[i];
        atomicAdd(&h[(int)mm.place(0.5f * r.xmin + 0.5f * r.xmax, 0)], 1u);
        atomicAdd(&h[AXIS_BINS + (int)mm.place(0.5f * r.ymin + 0.5f * r.ymax, 1)], 1u);
        atomicAdd(&h[2 * AXIS_BINS + (int)mm.place(0.5f * r.zmin + 0.5f * r.zmax, 2)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * AXIS_BINS; i += TPB)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// The share of the entries before every place (a warp per axis), and whether the order is that of x.
__global__ void k_axis_rank(const uint32_t *hist, uint64_t n, float *rank)
{
    if (threadIdx.x == 0)
        rank[3 * (AXIS_BINS + 1)] = n <= BY_X_ENTRIES * hist[3 * AXIS_BINS] ? 1.0f : 0.0f;
    const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
    constexpr int PER = AXIS_BINS / 32;
    uint32_t sum = 0;
    for (int k = 0; k < PER; k++) sum += hist[d * AXIS_BINS + lane * PER + k];
    uint32_t incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const float total = (float)max(1u, __shfl_sync(0xffffffffu, incl, 31));
    uint32_t run = incl - sum;
    float *r = rank + d * (AXIS_BINS + 1);
    for (int k = 0; k < PER; k++) {
        r[lane * PER + k] = (float)run / total;
        run += hist[d * AXIS_BINS + lane * PER + k];
    }
    if (lane == 31) r[AXIS_BINS] = 1.0f;
}

// Bounding record of every aligned chunk of 64 records, a warp per chunk.
__global__ void k_chunk_box(const Chunk *rec, uint64_t n, uint64_t nchunks, RecF *box)
{
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t c = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < nchunks;
         c += warps) {
        float lo[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
        float hi[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        for (int h = 0; h < 2; h++) {
            const uint64_t i = c * 64 + h * 32 + lane;
            if (i < n) {
                const RecF r = rec[c].r[h * 32 + lane];
                lo[0] = fminf(lo[0], r.xmin); hi[0] = fmaxf(hi[0], r.xmax);
                lo[1] = fminf(lo[1], r.ymin); hi[1] = fmaxf(hi[1], r.ymax);
                lo[2] = fminf(lo[2], r.zmin); hi[2] = fmaxf(hi[2], r.zmax);
                lo[3] = fminf(lo[3], r.t0); hi[3] = fmaxf(hi[3], r.t1);
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
#pragma unroll
            for (int k = 0; k < 4; k++) {
                lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
                hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
            }
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

// ---------------------------------------------------------------------------------------------
// temporal bins
// ---------------------------------------------------------------------------------------------
__global__ void k_bins_init(uint32_t m, double tmin, double b, double *bin_start,
                            unsigned long long *end_key)
{
    uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    bin_start[j] = part_bound(tmin, b, (int)j);
    end_key[j] = dkey(part_bound(tmin, b, (int)j + 1));
}

// off[j] = first sorted entry with bin >= j (bin_of is non-decreasing); *occupied (where asked for):
// bins with entries
__global__ void k_bin_bounds(const uint32_t *bin_of, uint64_t n, uint32_t m, uint32_t *off,
                             uint32_t *occupied)
{
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t j = s < n ? bin_of[s] : 0u;
    const uint32_t jp = s && s < n ? bin_of[s - 1] + 1 : 0u;
    const int heads = __syncthreads_count(s < n && jp <= j);
    if (threadIdx.x == 0 && heads && occupied) atomicAdd(occupied, (uint32_t)heads);
    if (s >= n) return;
    for (uint32_t k = jp; k <= j; k++) off[k] = (uint32_t)s;
    if (s == n - 1)
        for (uint32_t k = j + 1; k <= m; k++) off[k] = (uint32_t)n;
}

// The bins' ends and their prefix maximum (one block; maxima of the order keys).
__global__ void k_bin_ends(const unsigned long long *end_key, uint32_t m, double *bin_end,
                           double *pmax)
{
    __shared__ unsigned long long tot[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t per = (m + blockDim.x - 1) / blockDim.x;
    const uint32_t a = min(m, threadIdx.x * per), e = min(m, a + per);
    unsigned long long run = 0;
    for (uint32_t j = a; j < e; j++) run = max(run, end_key[j]);
    unsigned long long incl = run;  // prefix maximum over the threads
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl = max(incl, v);
    }
    if (lane == 31) tot[wid] = incl;
    __syncthreads();
    run = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) run = 0;
    for (int w = 0; w < wid; w++) run = max(run, tot[w]);
    for (uint32_t j = a; j < e; j++) {
        run = max(run, end_key[j]);
        bin_end[j] = dkey_inv(end_key[j]);
        pmax[j] = dkey_inv(run);
    }
}

// ---------------------------------------------------------------------------------------------
// partitions (subbins / grid)
// ---------------------------------------------------------------------------------------------
// Subbins per entry and dimension, in the sweep order `tid` of the bins' entries.
__global__ void k_part_count(const uint32_t *part_in, const uint32_t *orig, const uint32_t *tid,
                             uint64_t n, uint32_t *cnt)
{
    const uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t i = orig[tid[p]];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const uint32_t ab = part_in[(uint64_t)d * n + i];
        cnt[(uint64_t)d * n + p] = (ab >> 16) - (ab & 0xffffu) + 1u;
    }
}

__global__ void k_part_emit(const uint32_t *part_in, const uint32_t *orig, const uint32_t *tid,
                            uint64_t n, const uint32_t *pos, uint32_t *keys, uint32_t *vals)
{
    const uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t s = tid[p];
    const uint32_t ab = part_in[orig[s]];
    uint32_t at = pos[p];
    for (uint32_t j = ab & 0xffffu; j <= ab >> 16; j++, at++) {
        keys[at] = j;
        vals[at] = s;
    }
}

__global__ void k_st_hist(const uint32_t *keys, const uint32_t *ids, uint64_t len,
                          const uint32_t *bin_of, uint32_t m, uint32_t *cnt)
{
    uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= len) return;
    atomicAdd(&cnt[(uint64_t)keys[p] * m + bin_of[ids[p]]], 1u);
}

__global__ void k_gather_rec(const uint32_t *ids, uint64_t len, const RecF *rec, Chunk *out)
{
    uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= len) return;
    const uint32_t s = ids[p];
    out[p / CHUNK].r[p % CHUNK] = rec[s];
    out[p / CHUNK].id[p % CHUNK] = s;
}

// grid: every sorted entry is keyed by the cell of its MBB's minimum corner (single assignment)
__global__ void k_grid_key(const uint32_t *cell_in, const uint32_t *orig, uint64_t n, uint32_t *keys,
                           uint32_t *vals)
{
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    keys[s] = cell_in[orig[s]];
    vals[s] = (uint32_t)s;
}

__global__ void k_hist_u32(const uint32_t *keys, uint64_t len, uint32_t *cnt)
{
    uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < len) atomicAdd(&cnt[keys[p]], 1u);
}

int bits_for(uint64_t maxval)
{
    int b = 0;
    while (b < 64 && (maxval >> b) != 0) b++;
    return b;
}

struct Ctx {
    cudaStream_t s;
    DevBuf status;
    DevBuf rec;  // FP32 prefilter records in start-time order
    DevBuf tid;  // the bins' entries in their sweep order
    ts_status read_status()
    {
        uint32_t st = 0;
        TS_CUDA(cudaMemcpyAsync(&st, status.p, 4, cudaMemcpyDeviceToHost, s));
        TS_CUDA(cudaStreamSynchronize(s));
        if (st & DEV_ERR_INVALID) {
            set_error("invalid database segment (NaN/Inf or t_end <= t_start)");
            return TS_ERR_INVALID_ARG;
        }
        if (st & DEV_ERR_OVERFLOW) {
            set_error("index array longer than 2^32 - 1 entries");
            return TS_ERR_CAPACITY;
        }
        if (st) {
            set_error("index build: device status 0x%x", st);
            return TS_ERR_INTERNAL;
        }
        return TS_OK;
    }
};

// Bounding records of an array's chunks.
ts_status build_boxes(Ctx &c, Index *ix, const Chunk *rec, uint64_t n, RecF **box)
{
    const uint64_t nchunks = (n + 63) / 64;
    TS_CHECK(ix->alloc(box, nchunks));
    const unsigned cb = (unsigned)std::min<uint64_t>((nchunks * 32 + TPB - 1) / TPB, 152 * 32);
    if (nchunks) {
        k_chunk_box<<<cb, TPB, 0, c.s>>>(rec, n, nchunks, *box);
        TS_LAUNCHED();
    }
    return TS_OK;
}

// One dimension of the spatiotemporal index. The ids are emitted in the bins' sweep order and
// sorted stably by subbin, so a (subbin, bin) range keeps the Morton order inside and its chunks
// are small boxes too.
ts_status build_st_dim(Ctx &c, Index *ix, int dim, const uint32_t *part_in, const uint32_t *pos,
                       uint64_t len, const uint32_t *bin_of)
{
    const uint64_t n = ix->n;
    const int v = (int)ix->v[dim];
    DevBuf keys;
    TS_CHECK(keys.alloc(sizeof(uint32_t) * len, c.s));
    TS_CHECK(ix->alloc(&ix->st_ids[dim], len));
    k_part_emit<<<nblocks(n), TPB, 0, c.s>>>(part_in, ix->orig, c.tid.as<uint32_t>(), n, pos,
                                             keys.as<uint32_t>(), ix->st_ids[dim]);
    TS_LAUNCHED();
    TS_CHECK(radix_sort_u32(keys.as<uint32_t>(), ix->st_ids[dim], len, bits_for((uint64_t)v - 1),
                            c.s));
    uint64_t nbins = (uint64_t)v * ix->m;
    DevBuf h;
    TS_CHECK(h.alloc(sizeof(uint32_t) * nbins, c.s));
    TS_CUDA(cudaMemsetAsync(h.p, 0, sizeof(uint32_t) * nbins, c.s));
    k_st_hist<<<nblocks(len), TPB, 0, c.s>>>(keys.as<uint32_t>(), ix->st_ids[dim], len, bin_of,
                                             ix->m, h.as<uint32_t>());
    TS_LAUNCHED();
    TS_CHECK(ix->alloc(&ix->st_off[dim], nbins + 1));
    TS_CHECK(scan_u32(h.as<uint32_t>(), ix->st_off[dim], nbins, c.status.as<uint32_t>(), c.s));
    TS_CHECK(ix->alloc(&ix->st_rec[dim], (len + CHUNK - 1) / CHUNK));
    k_gather_rec<<<nblocks(len), TPB, 0, c.s>>>(ix->st_ids[dim], len, c.rec.as<RecF>(),
                                                ix->st_rec[dim]);
    TS_LAUNCHED();
    TS_CHECK(build_boxes(c, ix, ix->st_rec[dim], len, &ix->st_box[dim]));
    ix->st_len[dim] = len;
    return TS_OK;
}

ts_status build_grid(Ctx &c, Index *ix, const uint32_t *cell_in)
{
    const uint64_t n = ix->n;
    const int g = (int)ix->g;
    DevBuf keys;
    TS_CHECK(keys.alloc(sizeof(uint32_t) * n, c.s));
    TS_CHECK(ix->alloc(&ix->ga, n));
    k_grid_key<<<nblocks(n), TPB, 0, c.s>>>(cell_in, ix->orig, n, keys.as<uint32_t>(), ix->ga);
    TS_LAUNCHED();
    const uint64_t ncell = (uint64_t)g * g * g;
    TS_CHECK(radix_sort_u32(keys.as<uint32_t>(), ix->ga, n, bits_for(ncell - 1), c.s));
    DevBuf h;
    TS_CHECK(h.alloc(sizeof(uint32_t) * ncell, c.s));
    TS_CUDA(cudaMemsetAsync(h.p, 0, sizeof(uint32_t) * ncell, c.s));
    k_hist_u32<<<nblocks(n), TPB, 0, c.s>>>(keys.as<uint32_t>(), n, h.as<uint32_t>());
    TS_LAUNCHED();
    TS_CHECK(ix->alloc(&ix->g_off, ncell + 1));
    TS_CHECK(scan_u32(h.as<uint32_t>(), ix->g_off, ncell, c.status.as<uint32_t>(), c.s));
    TS_CHECK(ix->alloc(&ix->ga_rec, (n + CHUNK - 1) / CHUNK));
    k_gather_rec<<<nblocks(n), TPB, 0, c.s>>>(ix->ga, n, c.rec.as<RecF>(), ix->ga_rec);
    TS_LAUNCHED();
    // chunk bounding records: the cell sort is stable over the start-time order, so a chunk of
    // a cell spans a short stretch of time and a query's window skips most of a cell's chunks
    TS_CHECK(build_boxes(c, ix, ix->ga_rec, n, &ix->gbox));
    ix->g_len = n;
    return TS_OK;
}

}  // namespace

// What the freed indexes of a device may leave in the pool, all together: an index built in place of
// another of up to this size finds its memory mapped (1M segments, built, searched once and freed:
// 22 cudaMalloc and cudaFree took 1.6 of 3.5 ms).
constexpr size_t INDEX_KEEP = 512ull << 20;

void destroy_index(Index *ix)
{
    if (!ix) return;
    // On the index's own device, whichever the caller's is: freeing memory of a pool waits for
    // nothing, so whatever still reads the arrays has to have ended.
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != ix->device) cudaSetDevice(ix->device);
    cudaDeviceSynchronize();
    index_free(ix->allocs.data(), ix->allocs.size(), ix->bytes, INDEX_KEEP, ix->device);
    if (dev >= 0 && dev != ix->device) cudaSetDevice(dev);
    ix->magic = 0;
    delete ix;
}

// The partition's boundary table lo + j*w (j = 0..v), evaluated exactly as part_bound does.
static ts_status make_bounds(Index *ix, double **dst, double lo, double w, uint32_t v,
                             cudaStream_t s, PartTab *tab)
{
    TS_CHECK(ix->alloc(dst, v + 1));
    k_bounds<<<nblocks((uint64_t)v + 1), TPB, 0, s>>>(*dst, lo, w, v);
    TS_LAUNCHED();
    const float iw = w > 0.0 ? (float)(1.0 / w) : 0.0f;
    *tab = PartTab{*dst, lo, w, iw < 3.0e38f && w < 1.0e300 ? iw : 0.0f, (int)v};
    return TS_OK;
}

ts_status build_index(const ts_segments *db, const ts_index_params *p, cudaStream_t s,
                      Index **out)
{
    if (!db || !p || !out) {
        set_error("ts_build_index: NULL argument");
        return TS_ERR_INVALID_ARG;
    }
    *out = nullptr;
    if (db->n == 0 || db->n > 0x7fffffffull) {
        set_error("ts_build_index: database size %llu outside [1, 2^31 - 1]",
                  (unsigned long long)db->n);
        return TS_ERR_INVALID_ARG;
    }
    if (p->kind < TS_INDEX_BRUTE || p->kind > TS_INDEX_SPATIOTEMPORAL) {
        set_error("ts_build_index: unknown index kind %d", p->kind);
        return TS_ERR_INVALID_ARG;
    }
    if (p->grid_cells > 512) {
        set_error("ts_build_index: grid_cells %u above 512", p->grid_cells);
        return TS_ERR_INVALID_ARG;
    }
    const double *cols[8] = {db->x0, db->y0, db->z0, db->t0, db->x1, db->y1, db->z1, db->t1};
    for (int k = 0; k < 8; k++)
        if (!cols[k]) {
            set_error("ts_build_index: NULL column %d", k);
            return TS_ERR_INVALID_ARG;
        }
    const uint64_t n = db->n;
    Ctx c;
    c.s = s;
    TS_CHECK(c.status.alloc(4, s));
    TS_CUDA(cudaMemsetAsync(c.status.p, 0, 4, s));

    // device copy of the inputs when they live on the host
    DevBuf hostcopy;
    SegIn in;
    if (db->on_host) {
        TS_CHECK(hostcopy.alloc(sizeof(double) * n * 8, s));
        for (int k = 0; k < 8; k++) {
            double *dst = hostcopy.as<double>() + (uint64_t)k * n;
            TS_CUDA(cudaMemcpyAsync(dst, cols[k], sizeof(double) * n, cudaMemcpyHostToDevice, s));
            in.f[k] = dst;
        }
    } else {
        for (int k = 0; k < 8; k++) in.f[k] = cols[k];
    }

    Index *ix = new Index();
    ix->kind = p->kind;
    ix->n = n;
    ix->stream = s;
    cudaGetDevice(&ix->device);
    struct Guard {
        Index *&p;
        ~Guard() { if (p) destroy_index(p); }
    } guard{ix};

    // ingest
    DevBuf keys, vals, red;
    TS_CHECK(keys.alloc(sizeof(uint64_t) * n, s));
    TS_CHECK(vals.alloc(sizeof(uint32_t) * n, s));
    TS_CHECK(red.alloc(sizeof(unsigned long long) * R_N, s));
    k_init_red<<<1, 32, 0, s>>>(red.as<unsigned long long>());
    TS_LAUNCHED();
    k_ingest<<<std::min(nblocks(n), 152u * 8u), TPB, 0, s>>>(in, n, keys.as<uint64_t>(), vals.as<uint32_t>(),
                                        red.as<unsigned long long>(), c.status.as<uint32_t>());
    TS_LAUNCHED();
    unsigned long long hred[R_N];
    TS_CUDA(cudaMemcpyAsync(hred, red.p, sizeof(hred), cudaMemcpyDeviceToHost, s));
    TS_CHECK(c.read_status());
    ix->tmin = dkey_inv(hred[R_TMIN]);
    ix->tmax = dkey_inv(hred[R_TMAX]);
    ix->max_dur = dkey_inv(hred[R_DUR]);
    for (int d = 0; d < 3; d++) {
        ix->emin[d] = dkey_inv(hred[R_EMIN + d]);
        ix->emax[d] = dkey_inv(hred[R_EMAX + d]);
        ix->longest[d] = dkey_inv(hred[R_LONG + d]);
    }

    // temporal bins (all kinds: the schedule of every index starts from the time range)
    {
        uint64_t m = p->t_bins;
        double span = ix->tmax - ix->tmin;
        if (m == 0) {
            double mm = ix->max_dur > 0 ? ceil(4.0 * span / ix->max_dur) : 1.0;
            if (!(mm >= 1.0)) mm = 1.0;
            if (mm > (double)n) mm = (double)n;
            if (mm > 4e6) mm = 4e6;
            m = (uint64_t)mm;
        }
        if (p->kind == TS_INDEX_BRUTE || p->kind == TS_INDEX_SPATIAL) m = 1;
        if (m > 0x3fffffffull) {
            set_error("ts_build_index: t_bins %llu too large", (unsigned long long)m);
            return TS_ERR_INVALID_ARG;
        }
        ix->m = (uint32_t)m;
        ix->b = span / (double)ix->m;
    }
    // temporal bins, subbins (Sec. 4.3) or grid (Sec. 4.1): boundary tables, and the parts of every
    // entry
    DevBuf bin_in, part_in, bin_of, end_key;
    TS_CHECK(bin_in.alloc(sizeof(uint32_t) * n, s));
    TS_CHECK(bin_of.alloc(sizeof(uint32_t) * n, s));
    TS_CHECK(end_key.alloc(sizeof(unsigned long long) * ix->m, s));
    TS_CHECK(ix->alloc(&ix->bin_start, ix->m));
    TS_CHECK(ix->alloc(&ix->bin_end, ix->m));
    TS_CHECK(ix->alloc(&ix->bin_pmax, ix->m));
    TS_CHECK(ix->alloc(&ix->bin_off, (uint64_t)ix->m + 1));
    k_bins_init<<<nblocks(ix->m), TPB, 0, s>>>(ix->m, ix->tmin, ix->b, ix->bin_start,
                                               end_key.as<unsigned long long>());
    TS_LAUNCHED();
    PartTab bins{ix->bin_start, ix->tmin, ix->b,
                 ix->b > 0.0 && ix->b < 1.0e300 ? (float)(1.0 / ix->b) : 0.0f, (int)ix->m};
    if (!(bins.iw < 3.0e38f)) bins.iw = 0.0f;
    PartTab part[3] = {bins, bins, bins};
    if (p->kind == TS_INDEX_SPATIOTEMPORAL) {
        const uint32_t v_req = p->sub_bins ? p->sub_bins : 16u;
        for (int d = 0; d < 3; d++) {
            // v lowered so a subbin is at least as wide as the longest entry (Sec. 4.3)
            double ext = ix->emax[d] - ix->emin[d];
            double v = v_req < 1 ? 1.0 : (double)v_req;
            if (ix->longest[d] > 0.0) {
                double cap = floor(ext / ix->longest[d]);
                if (cap < 1.0) cap = 1.0;
                if (v > cap) v = cap;
            }
            if (!(ext > 0.0)) v = 1.0;
            if (v > 4096.0) v = 4096.0;
            ix->v[d] = (uint32_t)v;
            ix->sub_lo[d] = ix->emin[d];
            ix->sub_w[d] = ext / (double)ix->v[d];
            TS_CHECK(make_bounds(ix, &ix->sub_bound[d], ix->sub_lo[d], ix->sub_w[d], ix->v[d], s,
                                 &part[d]));
        }
        TS_CHECK(part_in.alloc(sizeof(uint32_t) * 3 * n, s));
    } else if (p->kind == TS_INDEX_SPATIAL) {
        const uint32_t g = p->grid_cells ? p->grid_cells : 50u;
        ix->g = g;
        for (int d = 0; d < 3; d++) {
            ix->g_lo[d] = ix->emin[d];
            ix->g_w[d] = (ix->emax[d] - ix->emin[d]) / (double)g;
            TS_CHECK(make_bounds(ix, &ix->g_bound[d], ix->g_lo[d], ix->g_w[d], g, s, &part[d]));
        }
        TS_CHECK(part_in.alloc(sizeof(uint32_t) * n, s));
    }
    k_parts<<<nblocks(n), TPB, 0, s>>>(in, n, bins, part[0], part[1], part[2], p->kind,
                                       bin_in.as<uint32_t>(), part_in.as<uint32_t>());
    TS_LAUNCHED();

    // sort by start time (stable: ties in input order), by the bits that vary
    TS_CHECK(radix_sort_u64(keys.as<uint64_t>(), vals.as<uint32_t>(), n, 64, s, nullptr, false,
                            hred[R_VARY]));
    TS_CHECK(ix->alloc(&ix->seg, n));
    TS_CHECK(c.rec.alloc(sizeof(RecF) * n, s));
    TS_CHECK(ix->alloc(&ix->orig, n));
    k_gather<<<nblocks(n), TPB, 0, s>>>(in, n, vals.as<uint32_t>(), bin_in.as<uint32_t>(), ix->seg,
                                        c.rec.as<RecF>(), ix->orig, bin_of.as<uint32_t>(),
                                        end_key.as<unsigned long long>());
    TS_LAUNCHED();
    keys.release();
    vals.release();
    DevBuf hist;  // entries by place (k_axis_hist), and the occupied bins
    if (p->kind != TS_INDEX_SPATIAL) {
        TS_CHECK(hist.alloc(sizeof(uint32_t) * (3 * AXIS_BINS + 1), s));
        TS_CUDA(cudaMemsetAsync(hist.p, 0, sizeof(uint32_t) * (3 * AXIS_BINS + 1), s));
    }
    k_bin_bounds<<<nblocks(n), TPB, 0, s>>>(bin_of.as<uint32_t>(), n, ix->m, ix->bin_off,
                                            hist.p ? hist.as<uint32_t>() + 3 * AXIS_BINS : nullptr);
    TS_LAUNCHED();
    k_bin_ends<<<1, 1024, 0, s>>>(end_key.as<unsigned long long>(), ix->m, ix->bin_end,
                                  ix->bin_pmax);
    TS_LAUNCHED();

    if (p->kind != TS_INDEX_SPATIAL) {
        // bins ordered along the Morton curve inside, or by x (ranges over the start-time order
        // cover whole bins): 4 bits an axis more than it takes to tell the entries of a mean bin apart
        const int per_bin = bits_for(n / ix->m);
        DevBuf tkeys;
        TS_CHECK(ix->alloc(&ix->axis_rank, 3 * (AXIS_BINS + 1) + 1));
        TS_CHECK(c.tid.alloc(sizeof(uint32_t) * n, s));
        const MortonMap mm =
            morton_map(ix, std::min(10, std::max(4, (per_bin + 2) / 3 + 4)));
        k_axis_hist<<<64, TPB, 0, s>>>(c.rec.as<RecF>(), n, std::max<uint64_t>(1, n >> 17), mm,
                                       hist.as<uint32_t>());
        TS_LAUNCHED();
        k_axis_rank<<<1, 96, 0, s>>>(hist.as<uint32_t>(), n, ix->axis_rank);
        TS_LAUNCHED();
        TS_CHECK(tkeys.alloc(sizeof(uint64_t) * n, s));
        k_tm_key<<<nblocks(n), TPB, 0, s>>>(c.rec.as<RecF>(), bin_of.as<uint32_t>(), n, mm,
                                            tkeys.as<uint64_t>(), c.tid.as<uint32_t>());
        TS_LAUNCHED();
        TS_CHECK(radix_sort_u64(tkeys.as<uint64_t>(), c.tid.as<uint32_t>(), n,
                                3 * mm.bits + bits_for((uint64_t)ix->m - 1), s, nullptr, false));
        TS_CHECK(ix->alloc(&ix->trec, (n + CHUNK - 1) / CHUNK));
        k_gather_rec<<<nblocks(n), TPB, 0, s>>>(c.tid.as<uint32_t>(), n, c.rec.as<RecF>(),
                                                ix->trec);
        TS_LAUNCHED();
        TS_CHECK(build_boxes(c, ix, ix->trec, n, &ix->tbox));
    }

    if (p->kind == TS_INDEX_SPATIOTEMPORAL) {
        // positions of the entries' ids in the three arrays; their lengths in one wait
        DevBuf cnt, pos;
        TS_CHECK(cnt.alloc(sizeof(uint32_t) * 3 * n, s));
        TS_CHECK(pos.alloc(sizeof(uint32_t) * 3 * (n + 1), s));
        k_part_count<<<nblocks(n), TPB, 0, s>>>(part_in.as<uint32_t>(), ix->orig,
                                                c.tid.as<uint32_t>(), n, cnt.as<uint32_t>());
        TS_LAUNCHED();
        uint32_t len[3];
        for (int d = 0; d < 3; d++) {
            uint32_t *pd = pos.as<uint32_t>() + d * (n + 1);
            TS_CHECK(scan_u32(cnt.as<uint32_t>() + d * n, pd, n, c.status.as<uint32_t>(), s));
            TS_CUDA(cudaMemcpyAsync(&len[d], pd + n, 4, cudaMemcpyDeviceToHost, s));
        }
        TS_CHECK(c.read_status());
        for (int d = 0; d < 3; d++)
            TS_CHECK(build_st_dim(c, ix, d, part_in.as<uint32_t>() + d * n,
                                  pos.as<uint32_t>() + d * (n + 1), len[d],
                                  bin_of.as<uint32_t>()));
    } else if (p->kind == TS_INDEX_SPATIAL) {
        TS_CHECK(build_grid(c, ix, part_in.as<uint32_t>()));
    }
    TS_CHECK(c.read_status());
    *out = ix;
    ix = nullptr;  // disarm the guard
    return TS_OK;
}

}  // namespace ts
