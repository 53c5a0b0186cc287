// ts_search.cu -- the search pipeline: query preparation and schedule, candidate units, groups,
// and the pair kernel with its count -> scan -> write result path.
//
// Paper mapping (Gowanlock & Casanova):
//   query preparation + schedule : the host-side schedule S of Sec. 4.2 and Sec. 4.3 and the
//                                  cell lookup of Sec. 4.1, here one device thread per query
//                                  segment (binary searches on the bins' prefix maximum replace
//                                  the carried scan; a dense cell offset array replaces the
//                                  binary search in G)
//   pair kernel                  : the compare() loop of Alg. 1-3. A warp takes a tile of up to
//                                  PK_TILE consecutive candidate records shared by a group of up
//                                  to 32 candidate ranges; each lane holds one record and the
//                                  warp loops over the group's members, so a record is fetched
//                                  once for up to 32 query segments. Results are counted,
//                                  scanned and written at fixed offsets instead of being appended
//                                  atomically to a fixed-size buffer.
//
// The pair test has three stages:
//   1. FP32 box test: time extents and the entry MBB against the query MBB expanded by d, all
//      bounds rounded outward (8 compares);
//   2. FP32 gap test: squared MBB distance accumulated rounding down against an upper bound of
//      d^2 (run only when some lane passed stage 1); a pair is dropped only when a lower bound
//      of its separation exceeds d, so no pair the FP64 test could accept is ever dropped;
//   3. the exact test on the survivors (the closed form of the interaction, in FP64 and in pairs of
//      FP32 values; ts_device.cuh), run 32 at a time on survivors compacted with ballot/popc.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <cstddef>
#include <mutex>
#include <vector>

#include "ts_device.cuh"
#include "ts_search.cuh"

namespace ts {

namespace {

constexpr int TPB = 256;
inline unsigned nblk(uint64_t n)
{
    uint64_t b = (n + TPB - 1) / TPB;
    if (b == 0) b = 1;
    if (b > 65535u * 32u) b = 65535u * 32u;
    return (unsigned)b;
}

// Relative slack added to the d-expanded query extents before they are mapped to subbins or grid
// cells, so FP64 rounding of (min - d) can never exclude a cell that holds a pair within d.
constexpr double EXT_SLACK = 1e-12;

__device__ __forceinline__ uint32_t req_of(const ReqDesc *reqs, uint32_t nreq, uint32_t i)
{
    uint32_t lo = 0, hi = nreq;  // last r with q_first <= i
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) / 2;
        if (reqs[mid].q_first <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Query preparation compares FP64 values by their order keys and rounds them to FP32 on the integer
// pipe; what is left to the FP64 pipe (2 lanes a clock and SM) are the velocities' divisions and the
// expanded extents. 800,000 query segments on the grid 194 -> 162 us, 100,000 on subbins 38 -> 31.
__device__ __forceinline__ bool finite_bits(double x)
{
    return ((uint32_t)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}

// x rounded to FP32 toward -inf (up = false) or +inf: truncated, and one step away from 0 when
// something was cut off on that side. Zero and what lies outside FP32's normal range: converted.
__device__ __forceinline__ float round_f32(double x, bool up)
{
    const long long u = dbits(x);
    const uint32_t hi = (uint32_t)((unsigned long long)u >> 32), lo = (uint32_t)u;
    if (((hi >> 20) & 0x7ffu) - 897u > 253u) return up ? __double2float_ru(x) : __double2float_rd(x);
    const uint32_t f = ((__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u) |
                       (hi & 0x80000000u);
    const bool away = (lo & 0x1fffffffu) != 0 && (u < 0) != up;
    return __uint_as_float(f + (away ? 1u : 0u));
}

__device__ __forceinline__ uint32_t first_pmax_above(const double *pmax, uint32_t m, uint64_t w0)
{
    uint32_t lo = 0, hi = m;
    while (lo < hi) {
        uint32_t mid = lo + (hi - lo) / 2;
        if (dkey(pmax[mid]) > w0) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// The part of x (as part_of) from the partition's boundary table bd[j] = lo + j*w: a first guess
// in FP32 (iwf ~ 1/w; 0 when w = 0), corrected by exact comparisons with the boundaries, so the
// result equals part_of's.
__device__ __forceinline__ int part_of_t(double x, const double *bd, float iwf, int v)
{
    const double lo = bd[0];
    const uint64_t kx = dkey(x);
    if (kx < dkey(lo)) return -1;
    if (v <= 1 || iwf == 0.0f) return v - 1;
    const float f = floorf((float)(x - lo) * iwf);
    int j = !(f < (float)v) ? v - 1 : (f < 0.0f ? 0 : (int)f);
    while (j + 1 < v && dkey(bd[j + 1]) <= kx) j++;
    while (j > 0 && dkey(bd[j]) > kx) j--;
    return j;
}

// First bin whose prefix maximum of B^end exceeds w0 (as first_pmax_above), searched in a bracket:
// pmax[j] >= B^start_{j+1} for every bin, so the answer is at most the bin holding w0 (jw); and
// since an entry lasts at most max_dur, bins more than `back` before jw are checked with one load
// (pmax[lo - 1] <= w0 keeps the answer at or after lo), otherwise the whole range is searched.
__device__ __forceinline__ uint32_t first_pmax_above_b(const double *pmax, const double *bs,
                                                       uint32_t m, float iwf, uint32_t back,
                                                       double w0)
{
    const int jw = part_of_t(w0, bs, iwf, (int)m);
    const uint64_t k0 = dkey(w0);
    if (jw < 0) return first_pmax_above(pmax, 1, k0);  // before every bin: 0 or (m = 1) 1
    uint32_t hi = (uint32_t)jw + 1 < m ? (uint32_t)jw + 1 : m;
    uint32_t lo = (uint32_t)jw > back ? (uint32_t)jw - back : 0u;
    if (lo > 0 && dkey(pmax[lo - 1]) > k0) lo = 0;
    // the answer lies in [lo, hi]; hi = m means no bin
    if (hi == m && !(dkey(pmax[m - 1]) > k0)) return m;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (dkey(pmax[mid]) > k0) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// last bin with start < w1, or -1 (the table lookup, then the strict comparison)
__device__ __forceinline__ int last_start_below_t(const double *bs, uint32_t m, float iwf,
                                                  double w1)
{
    int j = part_of_t(w1, bs, iwf, (int)m);
    const uint64_t k1 = dkey(w1);
    while (j >= 0 && !(dkey(bs[j]) < k1)) j--;
    return j;
}


// ---------------------------------------------------------------------------------------------
// query preparation (one thread per query segment of the batch)
// ---------------------------------------------------------------------------------------------
struct PrepParams {
    const double *f[8];
    uint64_t nq;
    int kind;
    const ReqDesc *reqs;
    uint32_t nreq;
    KeyFmt kf;
    MortonMap mm;  // of kf.morton bits per axis
    // index
    uint64_t n;
    uint32_t m;
    const double *bin_start, *bin_pmax;
    const uint32_t *bin_off;
    float bin_iwf;      // ~ 1 / bin width (first guesses only)
    uint32_t bin_back;  // bins an entry can reach back (from its duration), plus a margin
    uint32_t v[3];
    const double *sub_bound[3];  // subbin boundary tables (v + 1 each)
    float sub_iwf[3];
    const uint32_t *st_off[3];
    uint32_t g;
    const double *g_bound[3];    // grid boundary tables (g + 1 each)
    float g_iwf[3];
    double longest[3];
    uint32_t smem_bytes;  // > 0: the lookup tables are first copied into shared memory
    PipeBufs b;
};

// Sort key of a unit: (request, array, range start, Morton code of the query). Only the top
// lo_bits bits of the start are kept: the sort gathers units with nearby ranges, and among these
// near queries, into groups, and the groups order their members exactly before merging their
// ranges. (Grid units carry no code: their range is a run of cells near the query already.)
__device__ __forceinline__ uint64_t unit_key(uint32_t r, uint32_t sel, uint32_t lo, uint32_t code,
                                             KeyFmt f)
{
    const uint32_t sb = f.sel_bits ? (sel & ((1u << f.sel_bits) - 1u)) : 0u;
    const uint64_t k = ((uint64_t)r << (f.sel_bits + f.lo_bits)) | ((uint64_t)sb << f.lo_bits) |
                       (uint64_t)(lo >> f.lo_shift);
    return (k << (3 * f.morton)) | code;
}

// Lookup tables that k_qprep copies into shared memory: what the 48 KB a launch may ask for without
// an opt-in leave beside the kernel's own static arrays (the limit is on both together).
constexpr int QP_COUNTS = 2;
constexpr uint64_t QP_TABLE_BYTES = 48 * 1024 - QP_COUNTS * 32 * sizeof(uint32_t);

__global__ void k_qprep(PrepParams P)
{
    // the bin, subbin and cell boundary tables the lookups read, copied into shared memory (one
    // round of loads instead of chains of dependent global loads) when they fit; they belong to
    // the index, so the copy runs before the wait on the preceding kernel
    extern __shared__ __align__(16) unsigned char qp_smem[];
    const double *bin_start = P.bin_start, *bin_pmax = P.bin_pmax;
    const uint32_t *bin_off = P.bin_off;
    const double *sub_bound[3] = {P.sub_bound[0], P.sub_bound[1], P.sub_bound[2]};
    const double *g_bound[3] = {P.g_bound[0], P.g_bound[1], P.g_bound[2]};
    if (P.smem_bytes) {
        double *sd = reinterpret_cast<double *>(qp_smem);
        const uint32_t t = threadIdx.x, nt = blockDim.x;
        if (P.kind == TS_INDEX_SPATIAL) {
            for (int d = 0; d < 3; d++) {
                for (uint32_t i = t; i <= P.g; i += nt) sd[i] = P.g_bound[d][i];
                g_bound[d] = sd;
                sd += P.g + 1;
            }
        } else {
            for (uint32_t i = t; i < P.m; i += nt) sd[i] = P.bin_start[i];
            bin_start = sd;
            sd += P.m;
            for (uint32_t i = t; i < P.m; i += nt) sd[i] = P.bin_pmax[i];
            bin_pmax = sd;
            sd += P.m;
            if (P.kind == TS_INDEX_SPATIOTEMPORAL) {
                for (int d = 0; d < 3; d++) {
                    for (uint32_t i = t; i <= P.v[d]; i += nt) sd[i] = P.sub_bound[d][i];
                    sub_bound[d] = sd;
                    sd += P.v[d] + 1;
                }
            }
            uint32_t *so = reinterpret_cast<uint32_t *>(sd);
            for (uint32_t i = t; i <= P.m; i += nt) so[i] = P.bin_off[i];
            bin_off = so;
        }
        __syncthreads();
    }
    pdl_enter();
    const uint64_t nq = P.b.run ? min((uint64_t)P.b.run[0], P.nq) : P.nq;
    const uint32_t nreq = P.b.run ? P.b.run[1] : P.nreq;
    if (blockIdx.x == 0 && threadIdx.x == 0 && P.kind != TS_INDEX_SPATIAL)
        P.b.hdr[HDR_NU] = (uint32_t)nq;  // one unit slot per query
    uint32_t n_valid = 0, n_subbin = 0;  // (a warp's first active lane)
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nq;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = req_of(P.reqs, nreq, (uint32_t)i);
        const ReqDesc R = P.reqs[r];
        double v[8];
        bool fin = true;
        const uint64_t li = i - R.q_first;  // index within the request
#pragma unroll
        for (int k = 0; k < 8; k++) {
            v[k] = P.f[0] ? P.f[k][i] : R.cols[k][li];
            fin = fin && finite_bits(v[k]);
        }
        const bool ok = fin && dkey(v[7]) > dkey(v[3]);
        if (!ok) atomicOr(P.b.status, DEV_ERR_INVALID);
        const double dt = v[7] - v[3];
        QueryD q;
        q.vx = (v[4] - v[0]) / dt;
        q.vy = (v[5] - v[1]) / dt;
        q.vz = (v[6] - v[2]) / dt;
        q.w0 = dkey(v[3]) > dkey(R.t_start) ? v[3] : R.t_start;
        q.w1 = dkey(v[7]) < dkey(R.t_end) ? v[7] : R.t_end;
        const double dw = q.w0 - v[3];  // 0 unless the request interval clips the start
        q.xw = fma(q.vx, dw, v[0]);
        q.yw = fma(q.vy, dw, v[1]);
        q.zw = fma(q.vz, dw, v[2]);
        q.ndd = -R.dd;
        q.pad[0] = q.pad[1] = q.pad[2] = 0.0;
        const bool valid = ok && dkey(q.w0) < dkey(q.w1);
        P.b.qd[i] = q;
        P.b.qreq[i] = r;
        double mn[3], mx[3];
        float fmn[3], fmx[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const bool up = dkey(v[d]) < dkey(v[4 + d]);
            mn[d] = up ? v[d] : v[4 + d];
            mx[d] = up ? v[4 + d] : v[d];
            fmn[d] = round_f32(mn[d], false);
            fmx[d] = round_f32(mx[d], true);
        }
        P.b.qf[2 * i + 0] = make_float4(__fsub_rd(fmn[0], R.d_up), __fsub_rd(fmn[1], R.d_up),
                                        __fsub_rd(fmn[2], R.d_up), round_f32(q.w0, false));
        P.b.qf[2 * i + 1] = make_float4(__fadd_ru(fmx[0], R.d_up), __fadd_ru(fmx[1], R.d_up),
                                        __fadd_ru(fmx[2], R.d_up), round_f32(q.w1, true));

        uint32_t sel = SEL_T, lo = 0, hi = 0;
        bool subbin = false, unit = false;
        if (P.kind == TS_INDEX_SPATIAL) {
            // cells of the grid (single assignment by MBB minimum corner) that can hold an entry
            // within d: minimum corners in [min - d - longest, max + d] per axis
            uint32_t ca[3], cb[3];
            bool any = valid;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                double a = ((mn[d] - R.d) - P.longest[d]) -
                           EXT_SLACK * ((fabs(mn[d]) + R.d) + P.longest[d]);
                double bb = (mx[d] + R.d) + EXT_SLACK * (fabs(mx[d]) + R.d);
                int pa = part_of_t(a, g_bound[d], P.g_iwf[d], (int)P.g);
                int pb = part_of_t(bb, g_bound[d], P.g_iwf[d], (int)P.g);
                if (pa < 0) pa = 0;
                if (pb < pa) any = false;
                ca[d] = (uint32_t)pa;
                cb[d] = (uint32_t)(pb < 0 ? 0 : pb);
            }
            P.b.qcell[2 * i] = ca[0] | (ca[1] << 10) | (ca[2] << 20);
            P.b.qcell[2 * i + 1] = cb[0] | (cb[1] << 10) | (cb[2] << 20);
            P.b.qnu[i] = any ? (cb[0] - ca[0] + 1) * (cb[1] - ca[1] + 1) : 0u;
        } else {
            if (valid) {
                if (P.kind == TS_INDEX_BRUTE) {
                    hi = (uint32_t)P.n;
                } else {
                    // temporal range (Sec. 4.2 schedule)
                    const uint32_t jl = first_pmax_above_b(bin_pmax, bin_start, P.m,
                                                           P.bin_iwf, P.bin_back, q.w0);
                    const int jh = last_start_below_t(bin_start, P.m, P.bin_iwf, q.w1);
                    const bool any = (int)jl <= jh;
                    if (any) {
                        lo = bin_off[jl];
                        hi = bin_off[jh + 1];
                    }
                    if (any && P.kind == TS_INDEX_SPATIOTEMPORAL) {
                        // the dimension whose d-expanded extent meets one subbin (or none) with
                        // the fewest ids over the bins jl..jh (Sec. 4.3 schedule)
                        long long best = -1;
#pragma unroll
                        for (int d = 0; d < 3; d++) {
                            const int vv = (int)P.v[d];
                            double a = (mn[d] - R.d) - EXT_SLACK * (fabs(mn[d]) + R.d);
                            double bb = (mx[d] + R.d) + EXT_SLACK * (fabs(mx[d]) + R.d);
                            const int pa = part_of_t(a, sub_bound[d], P.sub_iwf[d], vv);
                            const int pb = part_of_t(bb, sub_bound[d], P.sub_iwf[d], vv);
                            const int ja = pa < 0 ? 0 : pa, jb = pb;
                            uint32_t clo, chi;
                            if (jb < ja) {
                                clo = 0;
                                chi = 0;
                            } else if (ja == jb) {
                                const uint32_t *off = P.st_off[d];
                                clo = off[(uint64_t)ja * P.m + jl];
                                chi = off[(uint64_t)ja * P.m + jh + 1];
                            } else {
                                continue;
                            }
                            if (best < 0 || (long long)(chi - clo) < best) {
                                best = (long long)(chi - clo);
                                sel = (uint32_t)d;
                                lo = clo;
                                hi = chi;
                            }
                        }
                        subbin = best >= 0;
                    }
                }
            }
            unit = valid && hi > lo;
            P.b.u_q[i] = (uint32_t)i;
            P.b.u_lo[i] = lo;
            P.b.u_hi[i] = hi;
            P.b.u_sel[i] = sel;
            const uint32_t code =
                P.kf.morton ? P.mm.code(0.5f * fmn[0] + 0.5f * fmx[0], 0.5f * fmn[1] + 0.5f * fmx[1],
                                        0.5f * fmn[2] + 0.5f * fmx[2])
                            : 0u;
            P.b.keys[i] = unit ? unit_key(r, sel, lo, code, P.kf) : ~0ull;
            P.b.vals[i] = (uint32_t)i;
        }
        const unsigned am = __activemask();
        const unsigned vm = __ballot_sync(am, valid);
        const unsigned sm = __ballot_sync(am, subbin);
        const int lane = threadIdx.x & 31;
        if (P.kind != TS_INDEX_SPATIAL) {
            // units per request: one atomic per request present in the warp (requests are
            // contiguous runs of queries, so nearly always one)
            const unsigned peers = __match_any_sync(am, r);
            const unsigned um = __ballot_sync(am, unit) & peers;
            if (um && lane == __ffs(peers) - 1) atomicAdd(&P.b.req_units[r], (uint32_t)__popc(um));
        }
        if (lane == __ffs(am) - 1) {
            n_valid += __popc(vm);
            n_subbin += __popc(sm);
        }
    }
    // the block's counts: one atomic per counter and block
    __shared__ uint32_t red[QP_COUNTS][32];
    const int warp = threadIdx.x >> 5, lane0 = threadIdx.x & 31;
    for (int o = 16; o; o >>= 1) {
        n_valid += __shfl_xor_sync(0xffffffffu, n_valid, o);
        n_subbin += __shfl_xor_sync(0xffffffffu, n_subbin, o);
    }
    if (lane0 == 0) {
        red[0][warp] = n_valid;
        red[1][warp] = n_subbin;
    }
    __syncthreads();
    if (threadIdx.x < QP_COUNTS) {
        unsigned long long v = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) v += red[threadIdx.x][w];
        if (v) atomicAdd(&P.b.stats[threadIdx.x == 0 ? ST_QSEGS : ST_SUBBIN], v);
    }
}

// Grid index: one unit per (cx, cy) of a query's cell box, covering cells cz_a..cz_b (a z-run
// of the row-major cell order, contiguous in the lookup array).
// One warp per 32 consecutive query segments: the lanes first load their query's cell box and
// unit slots (query i owns slots quoff[i] .. quoff[i] + qnu[i] - 1, so the warp's slots are one
// contiguous range), then run over the warp's slots 32 at a time, each lane finding the query of
// its slot among the lanes' starts; the unit counts per request are summed in the warp.
// all_or_none: more runs than the unit buffers hold leave no unit at all, and the kernels that
// follow nothing to do (a search in one go whose guess was too small starts over with exact sizes;
// what fits was sorted, swept and placed before: 60,000 queries of 20 cells on 100^3 cells
// 3,007 -> 2,618 us, 2,000 698 -> 511).
__global__ void k_grid_units(uint64_t nqcap, uint64_t ucap, KeyFmt kf, uint32_t g,
                             const uint32_t *g_off, bool all_or_none, PipeBufs b)
{
    pdl_enter();
    const unsigned FULL = 0xffffffffu;
    const uint64_t nq = b.run ? min((uint64_t)b.run[0], nqcap) : nqcap;
    if (all_or_none && b.quoff[nq] > ucap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) b.hdr[HDR_NU] = 0;
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        b.hdr[HDR_NU] = (uint32_t)min((uint64_t)b.quoff[nq], ucap);  // unit slots of the runs
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 32 < nq;
         w += warps) {
        const uint64_t i = w * 32 + lane;
        const bool has = i < nq;
        const uint32_t nu = has ? b.qnu[i] : 0u;
        // lanes past the last query start beyond every slot
        const uint32_t u0 = has ? b.quoff[i] : 0xffffffffu;
        const uint32_t r = has ? b.qreq[i] : 0u;
        const uint32_t c0 = has ? b.qcell[2 * i] : 0u, c1 = has ? b.qcell[2 * i + 1] : 0u;
        const int last = (int)min((uint64_t)31, nq - 1 - w * 32);
        const uint32_t ubeg = __shfl_sync(FULL, u0, 0);
        const uint32_t uend = __shfl_sync(FULL, u0 + nu, last);
        uint32_t cr = 0, cn = 0;  // this lane's running (request, valid units)
        for (uint32_t base = ubeg; base < uend; base += 32) {
            const uint32_t u = base + (uint32_t)lane;
            // the last lane whose start is at or before u owns slot u (a query without slots
            // shares its start with the next query, which then owns it)
            int j = 0;
#pragma unroll
            for (int step = 16; step; step >>= 1) {
                const uint32_t cand = __shfl_sync(FULL, u0, j + step);
                if (cand <= u) j += step;
            }
            const uint32_t ju0 = __shfl_sync(FULL, u0, j);
            const uint32_t jr = __shfl_sync(FULL, r, j);
            const uint32_t w0 = __shfl_sync(FULL, c0, j), w1 = __shfl_sync(FULL, c1, j);
            if (u >= uend) continue;
            if (u >= ucap) {  // more runs than the unit buffers hold
                atomicOr(b.status, DEV_ERR_OVERFLOW);
                continue;
            }
            const uint32_t ax = w0 & 1023u, ay = (w0 >> 10) & 1023u, az = (w0 >> 20) & 1023u;
            const uint32_t by = (w1 >> 10) & 1023u, bz = (w1 >> 20) & 1023u;
            const uint32_t ny = by - ay + 1;
            const uint32_t c = u - ju0;
            const uint32_t cx = ax + c / ny, cy = ay + c % ny;
            const uint64_t row = ((uint64_t)cx * g + cy) * g;
            const uint32_t lo = g_off[row + az], hi = g_off[row + bz + 1];
            b.u_q[u] = (uint32_t)(w * 32 + (uint64_t)j);
            b.u_lo[u] = lo;
            b.u_hi[u] = hi;
            b.u_sel[u] = SEL_GRID;
            b.keys[u] = hi > lo ? unit_key(jr, SEL_GRID, lo, 0u, kf) : ~0ull;
            b.vals[u] = u;
            if (jr != cr) {  // a request boundary inside the warp's slots (rare)
                if (cn) atomicAdd(&b.req_units[cr], cn);
                cr = jr;
                cn = 0;
            }
            cn += hi > lo;
        }
        // nearly always one request per warp: one atomic for the warp
        const uint32_t r0 = __shfl_sync(FULL, cr, 0);
        if (__all_sync(FULL, cr == r0 || cn == 0)) {
            uint32_t tot = cn;
            for (int o = 16; o; o >>= 1) tot += __shfl_xor_sync(FULL, tot, o);
            if (lane == 0 && tot) atomicAdd(&b.req_units[r0], tot);
        } else if (cn) {
            atomicAdd(&b.req_units[cr], cn);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// groups
// ---------------------------------------------------------------------------------------------
// Per request: unit starts (exclusive scan of its unit count) and group starts (ceil(units/32)).
// (With one request k_groups needs neither.)
__global__ void k_req_scan(uint32_t nreq_cap, PipeBufs b)
{
    pdl_enter();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const uint32_t nreq = b.run ? min(b.run[1], nreq_cap) : nreq_cap;
    uint32_t us = 0, gs = 0;
    for (uint32_t r = 0; r < nreq; r++) {
        b.ustart[r] = us;
        b.gstart[r] = gs;
        const uint32_t n = b.req_units[r];
        const uint32_t ng = (n + GROUP - 1) / GROUP;
        b.req_groups[r] = ng;
        us += n;
        gs += ng;
    }
    b.ustart[nreq] = us;
    b.gstart[nreq] = gs;
    b.hdr[HDR_U] = us;
    b.hdr[HDR_G] = gs;
}

// One warp per group: lane p holds the group's member p; the members are ordered by (array,
// start) with a bitonic network over the lanes, and their ranges (rounded down to chunks) are
// merged into disjoint segments (a member opens a segment when its start lies beyond every
// earlier range of its array); each segment is cut into tiles of `tile` records.
__global__ void k_groups(uint32_t nreq_cap, uint64_t gcap, uint32_t tile, const ReqDesc *reqs,
                         PipeBufs b)
{
    pdl_enter();
    // (also writes the members' records, in the group's order, for the pair kernel, and the bounds
    // of their boxes, against which k_tile_desc tests the chunks' bounding records)
    const unsigned FULL = 0xffffffffu;
    const uint32_t nreq = b.run ? min(b.run[1], nreq_cap) : nreq_cap;
    uint32_t G = b.hdr[HDR_G];
    if (nreq_cap == 1) {  // (what k_req_scan finds for several)
        const uint32_t nu = nreq ? b.req_units[0] : 0u;
        G = (nu + GROUP - 1) / GROUP;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            b.gstart[0] = 0;
            b.gstart[1] = G;
            b.hdr[HDR_U] = nu;
            b.hdr[HDR_G] = G;
        }
    }
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    unsigned long long n_cand = 0;  // candidates of this lane's members
    for (uint64_t g = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < gcap;
         g += warps) {
        if (g >= G) {
            if (lane == 0) b.ntiles[g] = 0;
            continue;
        }
        uint32_t r = 0, first = GROUP * (uint32_t)g, end = b.req_units[0];
        if (nreq_cap > 1) {
            uint32_t lo = 0, hi = nreq;  // last r with gstart[r] <= g
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) / 2;
                if (b.gstart[mid] <= g) lo = mid; else hi = mid;
            }
            r = lo;
            first = b.ustart[r] + GROUP * ((uint32_t)g - b.gstart[r]);
            end = b.ustart[r] + b.req_units[r];
        }
        end = min(first + GROUP, end);
        const uint32_t n = end - first;
        if (lane == 0) {
            const ReqDesc &R = reqs[r];
            b.ghdr[3 * g] =
                make_float4(R.d_dn, R.d2u, __uint_as_float(R.q_first), __uint_as_float(n));
        }
        // key = (array, start); lanes past the group's members hold the largest key
        uint64_t key = ~0ull;
        uint32_t mh = 0, mu = 0, cand = 0;
        if ((uint32_t)lane < n) {
            const uint32_t u = b.vals[first + lane];
            mu = u;
            const uint32_t us = b.u_sel[u];
            const uint32_t ul = b.u_lo[u];
            key = ((uint64_t)us << 32) | (ul & ~(uint32_t)(PK_CH - 1));  // chunk-aligned tiles
            mh = b.u_hi[u];
            cand = mh - ul;
        }
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                const uint64_t ok = __shfl_xor_sync(FULL, key, j);
                const uint32_t oh = __shfl_xor_sync(FULL, mh, j);
                const uint32_t ou = __shfl_xor_sync(FULL, mu, j);
                const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
                if (keep_min ? (ok < key) : (ok > key)) {
                    key = ok;
                    mh = oh;
                    mu = ou;
                }
            }
        }
        const bool member = (uint32_t)lane < n;
        const uint32_t sel = (uint32_t)(key >> 32), ml = (uint32_t)key;
        n_cand += cand;
        float4 ua = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        float4 ub = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (member) {
            MemberRec mr;
            mr.qi = b.u_q[mu];
            mr.lo = b.u_lo[mu];
            mr.hi = b.u_hi[mu];
            mr.sel = sel;
            mr.ea = b.qf[2 * (uint64_t)mr.qi + 0];
            mr.eb = b.qf[2 * (uint64_t)mr.qi + 1];
            b.gmem[(uint64_t)g * GROUP + lane] = mr;
            ua = mr.ea;
            ub = mr.eb;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            ua.x = fminf(ua.x, __shfl_xor_sync(FULL, ua.x, o));
            ua.y = fminf(ua.y, __shfl_xor_sync(FULL, ua.y, o));
            ua.z = fminf(ua.z, __shfl_xor_sync(FULL, ua.z, o));
            ua.w = fminf(ua.w, __shfl_xor_sync(FULL, ua.w, o));
            ub.x = fmaxf(ub.x, __shfl_xor_sync(FULL, ub.x, o));
            ub.y = fmaxf(ub.y, __shfl_xor_sync(FULL, ub.y, o));
            ub.z = fmaxf(ub.z, __shfl_xor_sync(FULL, ub.z, o));
            ub.w = fmaxf(ub.w, __shfl_xor_sync(FULL, ub.w, o));
        }
        if (lane < 2) b.ghdr[3 * g + 1 + lane] = lane ? ub : ua;
        // running maximum of the range ends over the earlier members of the same array
        uint32_t run = mh;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(FULL, run, o);
            const uint32_t vs = __shfl_up_sync(FULL, sel, o);
            if (lane >= o && vs == sel) run = max(run, v);
        }
        const uint32_t prev_run = __shfl_up_sync(FULL, run, 1);
        const uint32_t prev_sel = __shfl_up_sync(FULL, sel, 1);
        const bool start = member && (lane == 0 || prev_sel != sel || ml > prev_run);
        const unsigned starts = __ballot_sync(FULL, start);
        const unsigned nmask = n >= 32 ? FULL : ((1u << n) - 1u);
        const unsigned ends = n ? (((starts >> 1) | (1u << (n - 1))) & nmask) : 0u;
        // segment k ends at the lane before the next start (or at the last member)
        const bool is_end = n > 0 && ((ends >> lane) & 1u);
        const uint32_t a = 31 - __clz(starts & (lane == 31 ? FULL : ((2u << lane) - 1u)));
        const uint32_t seg_lo = __shfl_sync(FULL, ml, a & 31);
        const uint32_t ntile = is_end ? (run - seg_lo + tile - 1) / tile : 0u;
        uint32_t incl = ntile;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        if (is_end) {
            const uint32_t k = __popc(starts & (lane == 31 ? FULL : ((2u << lane) - 1u))) - 1;
            const uint64_t o = (uint64_t)g * GROUP + k;
            b.seg_lo[o] = seg_lo;
            b.seg_hi[o] = run;
            b.seg_sel[o] = sel;
            b.seg_t0[o] = incl - ntile;
        }
        if (lane == 31) {
            b.g_nseg[g] = __popc(starts);
            b.ntiles[g] = incl;
        }
    }
    // the block's candidates: one atomic per block
    __shared__ unsigned long long red[TPB / 32];
    for (int o = 16; o; o >>= 1) n_cand += __shfl_xor_sync(FULL, n_cand, o);
    if (lane == 0) red[threadIdx.x >> 5] = n_cand;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long v = 0;
        for (int w = 0; w < TPB / 32; w++) v += red[w];
        if (v) atomicAdd(&b.stats[ST_TESTS], v);
    }
}

__global__ void k_hdr(uint64_t gcap, uint64_t tcap, PipeBufs b)
{
    pdl_enter();
    const uint64_t T = b.tile_base[min((uint64_t)b.hdr[HDR_G], gcap)];
    b.hdr[HDR_T_LO] = (uint32_t)T;
    b.hdr[HDR_T_HI] = (uint32_t)(T >> 32);
    b.stats[ST_GROUPS] = b.hdr[HDR_G];
    b.stats[ST_TILES] = T;
    if (T > tcap || T > PK_MAX_TILES) atomicOr(b.status, DEV_ERR_OVERFLOW);
}

// The tiles that some member may meet, listed for the pair kernel (in no fixed order: a tile's rows
// are placed by its index) with the mask of their chunks whose bounding records meet the bounds
// of the group's members. Tiles and chunks that no member can meet cost a test here instead of a
// turn of a pair-kernel warp, and where tiles are many an entry holds a run of up to 32 chunks'
// tiles, so that a warp fetches the group's members once for all of them. `split` warps share a
// group's tiles, 32 tiles at a time. (1.13 G exact tests among 34M tiles of the grid: pair kernel
// 75.8 -> 68.0 ms with runs; where a warp gets fewer than 256 tiles, runs leave the last warps
// alone with long ones: 0.27 -> 0.31 ms on 180,000 tiles.)
//
// Listing tiles, ordering the temporal bins' entries and the queries along the Morton curve: the
// pair kernel on 100,000 merger query segments against 20M (temporal, d = 1) 2.42 -> 1.02 ms, on
// 50,000 dense ones against 2M (temporal, d = 2) 0.354 -> 0.23 ms. This kernel took 0.05 and
// 0.01 ms of it; it is bound by L2 latency (0.9 ms for 34M tiles of the grid).
__global__ void k_tile_desc(uint64_t gcap, uint64_t tcap, uint32_t tile, uint32_t pair_warps,
                            ArrayPtrs<const RecF> box, PipeBufs b)
{
    pdl_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0) b.stats[ST_CNT0] = globaltimer_ns();
    const uint32_t G = b.hdr[HDR_G];
    const uint64_t T = b.tile_base[min((uint64_t)G, gcap)];
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // the run header's tile count (as k_hdr)
        b.hdr[HDR_T_LO] = (uint32_t)T;
        b.hdr[HDR_T_HI] = (uint32_t)(T >> 32);
        b.stats[ST_GROUPS] = G;
        b.stats[ST_TILES] = T;
        if (T > tcap || T > PK_MAX_TILES) atomicOr(b.status, DEV_ERR_OVERFLOW);
    }
    if (T > tcap || T > PK_MAX_TILES) return;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    const uint64_t ngrp = min((uint64_t)G, gcap);
    const uint64_t split = max((uint64_t)1, warps / max((uint64_t)1, ngrp));
    const uint32_t tch = tile / PK_CH;
    // tiles per entry: as many as the 32 bits of its mask hold, but 256 tiles for every warp of
    // the pair kernel
    const uint32_t per = (uint32_t)max(1ull, min(32ull / tch, (unsigned long long)T / (256ull * pair_warps)));
    for (uint64_t k = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < ngrp * split;
         k += warps) {
        const uint64_t g = k / split;
        const uint32_t part = (uint32_t)(k % split);
        const uint64_t base = b.tile_base[g];
        const uint32_t ntile = (uint32_t)(b.tile_base[g + 1] - base);
        if (part * 32u >= ntile) continue;
        const uint32_t nseg = b.g_nseg[g];
        const float4 ua = b.ghdr[3 * g + 1], ub = b.ghdr[3 * g + 2];
        // lane k holds segment k (one round of loads for all the group's segments)
        uint32_t slo = 0, shi = 0, ssel = 0, st0 = 0xffffffffu;
        if ((uint32_t)lane < nseg) {
            const uint64_t o = (uint64_t)g * GROUP + lane;
            slo = b.seg_lo[o];
            shi = b.seg_hi[o];
            ssel = b.seg_sel[o];
            st0 = b.seg_t0[o];
        }
        for (uint32_t t0 = part * 32; t0 < ntile; t0 += (uint32_t)split * 32) {
            const uint32_t t = t0 + lane;
            // the last segment that starts at or before this lane's tile
            int j = 0;
#pragma unroll
            for (int step = 16; step; step >>= 1) {
                const uint32_t cand = __shfl_sync(FULL, st0, j + step);
                if (cand <= t) j += step;
            }
            const uint32_t lo = __shfl_sync(FULL, slo, j), hi = __shfl_sync(FULL, shi, j);
            const uint32_t sel = __shfl_sync(FULL, ssel, j), f = __shfl_sync(FULL, st0, j);
            uint32_t mask = 0, s0 = 0, nch = 0;
            const RecF *bx = nullptr;
            if (t < ntile) {
                s0 = lo + (t - f) * tile;
                bx = box.p[sel] + s0 / PK_CH;
                nch = min(tch, (hi - s0 + PK_CH - 1) / PK_CH);
                b.tile_hits[base + t] = 0;  // the count pass adds to it
            }
            // the 32 tiles' chunks, a lane per chunk: consecutive lanes read consecutive records
            for (uint32_t i = 0; i < tch; i++) {
                const uint32_t x = i * 32 + lane, l = x / tch, c = x - l * tch;
                const RecF *lbx = reinterpret_cast<const RecF *>(
                    __shfl_sync(FULL, reinterpret_cast<unsigned long long>(bx), l));
                const uint32_t ln = __shfl_sync(FULL, nch, l);
                const unsigned m = __ballot_sync(FULL, c < ln && filter_box(lbx[c], ua, ub));
                const int at = (int)(lane * tch) - (int)(i * 32);  // this lane's tile's first bit
                if (at > -32 && at < 32) mask |= at >= 0 ? m >> at : m << -at;
            }
            if (tch < 32) mask &= (1u << tch) - 1u;
            const uint32_t tmask = t < ntile ? mask : 0u;
            // one entry for a run of up to `per` tiles: its first tile's lane gathers their masks
            const uint32_t block = (uint32_t)j << 26 | (t - f) / per;  // (32 * 2^26 tiles)
            const uint32_t before = __shfl_up_sync(FULL, block, 1);
            const bool head = t < ntile && (lane == 0 || before != block);
            for (uint32_t k = 1; k < per; k++) {
                const uint32_t m = __shfl_down_sync(FULL, tmask, k);
                const uint32_t o = __shfl_down_sync(FULL, block, k);
                if (lane + k < 32 && o == block) mask |= m << (k * tch);
            }
            const unsigned any = __ballot_sync(FULL, head && mask != 0u);
            uint32_t at = 0;
            if (lane == 0 && any) at = atomicAdd(&b.counters[2], (uint32_t)__popc(any));
            at = __shfl_sync(FULL, at, 0);
            if (head && mask)
                b.tdesc[at + __popc(any & ((1u << lane) - 1u))] =
                    make_uint4((uint32_t)(base + t) | (sel << 29), mask, (uint32_t)g, s0);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// pair kernel
// ---------------------------------------------------------------------------------------------
struct __align__(16) WarpSmem {
    Chunk stage[PK_STAGES];
    MemberRec mem[GROUP];  // the tile's group members
    float4 ghdr;           // their request's d_dn, d2u, q_first, and their number
    uint4 dnext;           // the next listed tile (asynchronous copy during the sweep)
    RecF cbox[32];         // bounding records of the tile's chunks
    // exact-test queue, first in first out, carried from tile to tile: query index in the batch,
    // entry, tile, query index within its request
    uint32_t q_qi[PK_QUEUE], q_e[PK_QUEUE], q_tile[PK_QUEUE], q_ql[PK_QUEUE];
    uint32_t plist[PK_PLIST];  // (member << 8 | slot) pairs of a chunk that passed the box test
    unsigned long long bar[PK_STAGES];
    unsigned long long mbar;  // members + chunk boxes
    unsigned long long xbar;  // injected stall (tests): a barrier nothing ever arrives on
    // counts: chunks, bitmask chunks, sparse member visits, survivors, exact tests, hits
    unsigned long long count[6];
    uint32_t wt_cur, wt_cnt;  // last tile with hits, its hits so far
    // Count pass: this warp's part [sc_at, sc_end) of the scratch. Parts are taken from a shared
    // counter, 32 slots first and then half of what the warp has had (sc_had), at most 256: an
    // atomic for every batch of hits put its round trip to L2 into each batch, and all of them on
    // one address. `room` until a part did not fit.
    uint32_t sc_at, sc_end, sc_had, room;
};

enum { PASS_COUNT = 0, PASS_WRITE = 1 };

// Flag beside a tile's hit count, set by the count pass on a tile with a hit that the scratch did
// not keep: the write pass sweeps exactly the flagged tiles (k_place writes the rows of the kept
// hits, the same rows the sweep gives them). A tile has at most 2048 x 32 hits.
constexpr uint32_t TILE_REDO = 0x80000000u;

struct PairParams {
    PipeBufs b;
    const Chunk *rec[5];
    const RecF *box[5];  // bounding record per chunk
    const SegD *seg;
    const uint32_t *orig;
    uint64_t tcap;
    uint64_t rows_cap;  // write pass: rows beyond this capacity are not written (flagged)
    uint64_t scap;      // slots for the hits that the count pass keeps for placement
    bool exact_parts;   // warps take as many slots as they have hits, none in advance
    uint32_t tile;      // records per tile
    uint32_t tile_inv;  // ceil(2^16 / chunks per tile): c * it >> 16 is chunk c's tile (c < 32)
    // > 0 (tests only): the first warp of block 0 waits this long on a barrier phase that never
    // completes before taking any tile, so the kernel's timeout path runs (status, return)
    uint64_t stall_ns;
};

// Exact test of nflush queued candidates from the queue's place `at` on, one per lane, and what
// becomes of their hits.
template <int PASS>
__device__ __forceinline__ void pair_batch(WarpSmem &W, const PairParams &P, uint32_t at,
                                           uint32_t nflush)
{
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const PipeBufs &B = P.b;
    uint32_t qi = 0, eid = 0, tile = 0xffffffffu, ql = 0, orig = 0;
    if ((uint32_t)lane < nflush) {
        qi = W.q_qi[at + lane];
        eid = W.q_e[at + lane];
        tile = W.q_tile[at + lane];
        ql = W.q_ql[at + lane];
        orig = P.orig[eid];
    }
    const bool room = W.room != 0;
    // the count pass computes hit intervals only while the scratch still has room, as far as this
    // warp has seen (after an overflow the write pass sweeps and computes them)
    const bool interval = PASS == PASS_WRITE || room;
    bool h = false;
    double tin = 0.0, tout = 0.0;
    if ((uint32_t)lane < nflush) {
        SegD e;
        QueryD q;
        ld32(P.seg + eid, &e.x0);
        ld32(&P.seg[eid].vx, &e.vx);
        ld32(B.qd + qi, &q.xw);
        ld32(&B.qd[qi].vx, &q.vx);
        q.ndd = B.qd[qi].ndd;
        h = pair_test(q, e, interval, &tin, &tout);
    }
    const unsigned hm = __ballot_sync(FULL, h);
    if (lane == 0) {
        W.count[4] += nflush;
        W.count[5] += __popc(hm);
    }
    if (!hm) return;
    // hits of the same tile (the queue holds a tile's candidates contiguously, tiles in the order
    // this warp took them)
    const unsigned mine = hm & __match_any_sync(FULL, h ? tile : 0xffffffffu);
    // rank of the hit among its tile's rows (queue order, the same in both passes)
    const uint32_t wt_cur = W.wt_cur, wt_cnt = W.wt_cnt;
    const uint32_t rank = (tile == wt_cur ? wt_cnt : 0u) + __popc(mine & lt_mask);
    if (PASS == PASS_COUNT) {
        if (h && (mine & lt_mask) == 0) atomicAdd(&B.tile_hits[tile], (uint32_t)__popc(mine));
        const uint32_t sc_at = W.sc_at, sc_end = W.sc_end;
        const uint32_t nh = __popc(hm), left = sc_end - sc_at;
        const uint32_t k = __popc(hm & lt_mask);  // rank among the batch's hits
        uint32_t slot = sc_at + k;
        bool kept = h && k < left;
        __syncwarp();
        if (nh <= left) {
            if (lane == 0) W.sc_at = sc_at + nh;
        } else if (room) {
            const uint32_t had = W.sc_had;
            const uint32_t want = P.exact_parts ? nh - left : min(256u, max(32u, had / 2));
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(&B.stats[ST_SCRATCH], (unsigned long long)want);
            base = __shfl_sync(FULL, base, 0);
            if (base + want <= P.scap) {
                if (k >= left) slot = (uint32_t)base + (k - left);
                kept = h;
                if (lane == 0) {
                    W.sc_at = (uint32_t)base + (nh - left);
                    W.sc_end = (uint32_t)base + want;
                    W.sc_had = had + want;
                }
            } else {
                // (the part's slots inside the scratch hold no hit)
                for (unsigned long long j = base + lane; j < P.scap; j += 32)
                    B.s_tile[j] = 0xffffffffu;
                if (lane == 0) {
                    B.stats[ST_LOST] = 1;
                    W.sc_at = sc_end;
                    W.room = 0;
                }
            }
        }
        if (kept) {
            B.s_tile[slot] = tile;
            B.s_rank[slot] = rank;
            B.s_q[slot] = ql;
            B.s_e[slot] = orig;
            B.s_tin[slot] = tin;
            B.s_tout[slot] = tout;
        }
        // a tile with a hit the scratch could not keep is swept again by the write pass
        const unsigned lost = __ballot_sync(FULL, h && !kept);
        if (h && !kept && (mine & lost & lt_mask) == 0)
            atomicOr(&B.tile_hits[tile], TILE_REDO);
    } else if (h) {
        const uint64_t o = B.tile_off[tile] + rank;
        if (o < B.tile_off[tile + 1]) {
            B.out_q[o] = ql;
            B.out_e[o] = orig;
            B.out_tin[o] = tin;
            B.out_tout[o] = tout;
        } else {
            atomicOr(B.status, DEV_ERR_INTERNAL);  // the passes disagree
        }
    }
    const int last = 31 - __clz(hm);
    const uint32_t last_tile = __shfl_sync(FULL, tile, last);
    const uint32_t last_n = __popc(__shfl_sync(FULL, mine, last));
    __syncwarp();
    if (lane == 0) {
        W.wt_cnt = (last_tile == wt_cur ? wt_cnt : 0u) + last_n;
        W.wt_cur = last_tile;
    }
    __syncwarp();
}

// Exact tests of the queued candidates, oldest first, 32 at a time; with `all` the rest too.
// Returns how many stay queued (moved to the front). Not inlined, and called only between two
// chunks' survivors and at a warp's end, where the sweep has little in registers (what lasts is in
// shared memory), so that those of the exact test do not limit the warps that sweep.
template <int PASS>
__device__ __noinline__ uint32_t pair_flush(uint32_t qn, bool all)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    WarpSmem &W = reinterpret_cast<WarpSmem *>(smem_raw)[threadIdx.x >> 5];
    const PairParams &P = *reinterpret_cast<const PairParams *>(smem_raw + PK_WARPS * sizeof(WarpSmem));
    const int lane = threadIdx.x & 31;
    uint32_t at = 0;
    __syncwarp();
    for (; qn - at >= 32; at += 32) pair_batch<PASS>(W, P, at, 32);
    if (all && qn > at) {
        pair_batch<PASS>(W, P, at, qn - at);
        at = qn;
    }
    uint32_t v[4];
    const bool keep = at + lane < qn;
    if (keep) {
        v[0] = W.q_qi[at + lane];
        v[1] = W.q_e[at + lane];
        v[2] = W.q_tile[at + lane];
        v[3] = W.q_ql[at + lane];
    }
    __syncwarp();
    if (keep) {
        W.q_qi[lane] = v[0];
        W.q_e[lane] = v[1];
        W.q_tile[lane] = v[2];
        W.q_ql[lane] = v[3];
    }
    __syncwarp();
    return qn - at;
}

// Persistent pair kernel. Warps take listed tiles (a group of up to 32 query units and up to
// `tile` consecutive entries of one sorted array, or a run of such tiles): the first by their
// index in the grid, the rest from a device counter. Entry records stream through a ring of
// PK_STAGES shared-memory buffers filled by 1-D bulk copies. The conservative FP32 filters pick the
// candidates of the exact test; those wait in a per-warp queue that is carried across tiles and
// drained 32 at a time, so that the exact tests run on full warps.
//
// Bound: instruction issue (63 % of the slots on 11 M exact tests among 2.3 G candidates; ALU 50 %,
// shared-memory wavefronts 52 %, FP64 33 %). What it waits for is mostly the fixed latency of its
// own arithmetic, so the number of resident warps counts: 20 per SM (96 registers) instead of 16
// took 1.13 G exact tests (merger, 20M segments, d = 1 and 5) from 88 to 76 ms; 24 (80
// registers, spilled, and little L1 left) take 122. Flushes where the queue fills, rather than
// in the middle of every batch of survivors, the ids beside the records and the scratch taken in
// parts: 100 to 88 ms. Count pass: hits per tile. Write pass: the rows of every
// tile with hits, at its offset from the scan, in queue order (the same order in both passes, so
// the offsets match).
template <int PASS>
__global__ void __launch_bounds__(PK_THREADS, PK_MIN_BLOCKS) k_pair(const PairParams P)
{
    pdl_enter();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // (pair_flush's copy of the parameters)
    if (threadIdx.x == 0)
        *reinterpret_cast<PairParams *>(smem_raw + PK_WARPS * sizeof(WarpSmem)) = P;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    WarpSmem &W = reinterpret_cast<WarpSmem *>(smem_raw)[wid];
    const unsigned FULL = 0xffffffffu;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const PipeBufs &B = P.b;

    if (lane == 0) {
        for (int k = 0; k < 6; k++) W.count[k] = 0;
        W.wt_cur = 0xffffffffu;
        W.wt_cnt = 0;
        W.sc_at = W.sc_end = W.sc_had = 0;
        W.room = PASS == PASS_COUNT;
        for (int k = 0; k < PK_STAGES; k++) mbar_init(&W.bar[k], 1);
        mbar_init(&W.mbar, 1);
        mbar_init(&W.xbar, 1);
        fence_mbar_init();
    }
    __syncwarp();
    // bits k: the parity the next wait on bar[k] is for, bit PK_STAGES: on mbar; and the copies in
    // flight
    uint32_t parity = 0u, pending = 0u;
    constexpr uint32_t MEM = 1u << PK_STAGES;
    bool abort = false;
    if (P.stall_ns && blockIdx.x == 0 && wid == 0)
        abort = !mbar_wait_bounded(&W.xbar, 0u, P.stall_ns);  // (never arrived on: times out)

    const uint64_t all_tiles = (uint64_t)B.hdr[HDR_T_LO] | ((uint64_t)B.hdr[HDR_T_HI] << 32);
    uint32_t ntiles = B.counters[2];  // listed tiles
    if (all_tiles > P.tcap || all_tiles > PK_MAX_TILES) ntiles = 0;  // overflow already flagged
    if (PASS == PASS_WRITE && B.stats[ST_LOST] == 0)
        ntiles = 0;  // the count pass kept every hit: k_place writes the rows
    // (otherwise the write pass sweeps only the tiles whose hits were not all kept)
    if (PASS == PASS_WRITE && ntiles && B.tile_off[all_tiles] > P.rows_cap) {
        // more rows than the output holds: write none (the caller sees the exact count)
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(B.status, DEV_ERR_OVERFLOW);
        ntiles = 0;
    }
    uint32_t qn = 0;  // queued candidates (warp-uniform)

    // listed tiles are taken from a device counter; the next entry is fetched while a tile is
    // swept
    // (each warp's first tile is its index in the grid, so the counter only hands out the rest:
    // no burst of same-address atomics when every warp starts at once)
    const uint32_t nwarps = gridDim.x * PK_WARPS;
    uint32_t t = blockIdx.x * PK_WARPS + wid;
    uint4 D = t < ntiles ? B.tdesc[t] : make_uint4(0u, 0u, 0u, 0u);
    while (!abort && t < ntiles) {
        uint32_t t_next = 0;
        if (lane == 0) t_next = nwarps + atomicAdd(&B.counters[PASS], 1u);
        if (PASS == PASS_WRITE) {
            // the chunks of the entry's tiles that have rows the count pass did not keep
            const uint32_t tch = P.tile / PK_CH, c = (uint32_t)lane * tch;
            bool redo = false;
            if (c < 32 && (D.y >> c) != 0u) {  // (a tile of the entry, or before its last one)
                const uint32_t th = B.tile_hits[(D.x & PK_MAX_TILES) + lane];
                redo = (th & TILE_REDO) != 0;
            }
            const uint32_t bits = tch < 32 ? (1u << tch) - 1u : FULL;
            D.y &= __reduce_or_sync(FULL, redo ? bits << c : 0u);
            if (!D.y) {
                t = __shfl_sync(FULL, t_next, 0);
                D = t < ntiles ? B.tdesc[t] : make_uint4(0u, 0u, 0u, 0u);
                continue;
            }
        }
        const uint32_t tile0 = D.x & PK_MAX_TILES, sel = D.x >> 29, cand = D.y, s0 = D.w;
        // the chunk at s0 + c * PK_CH, whole (slots past the array's end or a member's range are
        // masked by the range)
        auto copy_chunk = [&](uint32_t c, uint32_t st) {
            mbar_arrive_tx(&W.bar[st], (uint32_t)sizeof(Chunk));
            bulk_g2s(&W.stage[st], P.rec[sel] + s0 / PK_CH + c, (uint32_t)sizeof(Chunk), &W.bar[st]);
        };
        // one bulk copy of the members and of the chunks' bounding records, then the first two
        // listed chunks of records
        uint32_t pend = cand, first = 0;
        if (lane == 0) {
            const uint32_t g = D.z;
            const uint32_t mb = GROUP * (uint32_t)sizeof(MemberRec);
            const uint32_t cb = (32 - __clz(cand)) * (uint32_t)sizeof(RecF);
            mbar_arrive_tx(&W.mbar, mb + cb + (uint32_t)sizeof(float4));
            bulk_g2s(&W.ghdr, B.ghdr + 3 * (uint64_t)g, (uint32_t)sizeof(float4), &W.mbar);
            bulk_g2s(&W.mem[0], B.gmem + (uint64_t)g * GROUP, mb, &W.mbar);
            bulk_g2s(&W.cbox[0], P.box[sel] + s0 / PK_CH, cb, &W.mbar);
        }
        pending = MEM;
#pragma unroll
        for (int k = 0; k < PK_STAGES; k++) {
            if (pend) {
                if (lane == 0) copy_chunk(__ffs(pend) - 1, k);
                pending |= 1u << k;
                first |= pend & (0u - pend);
                pend &= pend - 1u;
            }
        }
        if (!mbar_wait_bounded(&W.mbar, (parity >> PK_STAGES) & 1u)) {
            abort = true;
            break;
        }
        parity ^= MEM;
        pending &= ~MEM;
        // the next tile's entry is copied into shared memory during the sweep
        if (lane == 0 && t_next < ntiles) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(&W.dnext)),
                         "l"(B.tdesc + t_next)
                         : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        // the listed chunks this lane's member meets: its range overlaps the chunk and its
        // expanded box meets the chunk's bounding record
        uint32_t mc = 0u;
        if ((uint32_t)lane < __float_as_uint(W.ghdr.w) && W.mem[lane].sel == sel) {
            const MemberRec M = W.mem[lane];
            for (uint32_t rem = cand; rem; rem &= rem - 1u) {
                const uint32_t c = __ffs(rem) - 1;
                const uint32_t cs = s0 + c * PK_CH, ce = cs + PK_CH;
                const bool meet = (M.lo < ce) & (M.hi > cs) & filter_box(W.cbox[c], M.ea, M.eb);
                mc |= (uint32_t)meet << c;
            }
        }
        __syncwarp();

        // a candidate that passed the filters joins the exact-test queue; its exact record, a
        // gather from HBM, is on its way to L2 while it waits there
        uint32_t tile = tile0;  // (of the chunk being swept)
        auto enqueue = [&](bool p, uint32_t qi, uint32_t e) {
            const unsigned bm = __ballot_sync(FULL, p);
            if (bm) {
                if (p) {
                    const uint32_t j = qn + __popc(bm & lt_mask);
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(P.seg + e));
                    W.q_qi[j] = qi;
                    W.q_e[j] = e;
                    W.q_tile[j] = tile;
                    W.q_ql[j] = qi - __float_as_uint(W.ghdr.z);
                }
                qn += __popc(bm);
            }
        };

        // chunks to sweep, in order; the first PK_STAGES listed ones were copied already, later
        // ones are copied PK_STAGES sweeps ahead, so of these a chunk no member meets is neither
        // copied nor swept
        const uint32_t need = __reduce_or_sync(FULL, mc);
        uint32_t todo = need | first;
        pend &= need;
        for (uint32_t st = 0; todo; st = st + 1 == PK_STAGES ? 0 : st + 1) {
            const uint32_t c = __ffs(todo) - 1;
            todo &= todo - 1u;
            if (!mbar_wait_bounded(&W.bar[st], (parity >> st) & 1u)) {
                abort = true;
                break;
            }
            parity ^= 1u << st;
            pending &= ~(1u << st);
            if (PASS == PASS_COUNT && lane == 0) W.count[0]++;
            const Chunk &C = W.stage[st];
            tile = tile0 + ((c * P.tile_inv) >> 16);
            const unsigned act = __ballot_sync(FULL, (mc >> c) & 1u);
            // what is left of the chunk: members of the per-member pass, listed pairs [b, npl),
            // survivors of the bitmask pass (none of them when no member meets a chunk that was
            // copied ahead of the member tests)
            unsigned rem = act;
            uint32_t npl = 0, b = 0, m0 = 0u, m1 = 0u;
            if (sel == SEL_GRID && __popc(act) > PK_SPARSE) {
                rem = 0u;
                if (PASS == PASS_COUNT && lane == 0) W.count[1]++;
                // stage 1: two axes of every slot against every member (slot i is read at a
                // warp-uniform address, a shared-memory broadcast); bit i is set when the extents
                // overlap on both. 16 slots at a time and two accumulators: unrolled further, the
                // loads in flight take the registers of more warps. Time and x: a cell holds
                // entries of every time.
                //
                // Only for the grid's cells. The other arrays' chunks are small boxes within one
                // bin, which most survivors of two axes miss on the third: the per-member pass
                // tests all at once and lists what is left for full warps (100,000 merger
                // queries, temporal, d = 1: 1.05 ms with this pass above 8 members, 0.74 above 16,
                // 0.69 without; dense plan 0.27, 0.22, 0.215).
                const MemberRec &M = W.mem[lane];
                const float fa = M.ea.w, fb = M.eb.w, ga = M.ea.x, gb = M.eb.x;
                const float2 *ax = reinterpret_cast<const float2 *>(&C.r[0]) + 3;
                const float2 *ax2 = reinterpret_cast<const float2 *>(&C.r[0]);
#pragma unroll 1
                for (int j = 0; j < 4; j++) {
                    uint32_t a[2] = {0u, 0u};
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const float2 v = ax[64 * j + 4 * i], u = ax2[64 * j + 4 * i];
                        if ((v.y >= fa) & (v.x <= fb) & (u.y >= ga) & (u.x <= gb))
                            a[i & 1] |= 1u << i;
                    }
                    m0 = (m0 >> 16) | (m1 << 16);  // the 64 bits move down, these join on top
                    m1 = (m1 >> 16) | ((a[0] | a[1]) << 16);
                }
                // this lane's own range within the chunk, as bits of the 64 slots
                const uint32_t cs = s0 + c * PK_CH;
                const uint32_t x = max(M.lo, cs) - cs, y = min(M.hi - cs, (uint32_t)PK_CH);
                if ((act >> lane) & 1u) {
                    m0 &= (y >= 32 ? FULL : ((1u << y) - 1u)) & (x >= 32 ? 0u : (FULL << x));
                    m1 &= y <= 32 ? 0u : ((y >= 64 ? FULL : ((1u << (y - 32)) - 1u)) &
                                          (x <= 32 ? FULL : (FULL << (x - 32))));
                } else {
                    m0 = m1 = 0u;
                }
            } else if (PASS == PASS_COUNT && lane == 0) {
                W.count[2] += __popc(act);
            }
            for (bool more = true; more;) {
                while (qn <= PK_QUEUE - 32) {
                    bool p = false;
                    uint32_t qi = 0, e = 0;
                    if (b < npl) {
                        // the listed pairs go through the gap bound one per lane, so that the gap
                        // bound and the queue run on full warps
                        if (b + lane < npl) {
                            const uint32_t x = W.plist[b + lane];
                            const MemberRec &M = W.mem[x >> 8];
                            qi = M.qi;
                            e = C.id[x & 63u];
                            p = filter_gap_e(C.r[x & 63u], M.ea, M.eb, W.ghdr.x, W.ghdr.y);
                        }
                        b += 32;
                    } else if (rem) {
                        // few members meet this chunk: one lane per slot (slots lane and lane +
                        // 32), the members that meet the chunk in turn, their boxes read as
                        // broadcasts; the (member, slot) pairs that pass the box test are listed
                        // in shared memory (member by member, slot order)
                        __syncwarp();
                        const uint32_t pos = s0 + c * PK_CH + lane;
                        const RecF r0 = C.r[lane], r1 = C.r[lane + 32];
                        npl = b = 0;
                        // (room for one more member's 64 pairs)
                        for (; rem && npl <= PK_PLIST - 64; rem &= rem - 1u) {
                            const uint32_t m = __ffs(rem) - 1;
                            const MemberRec &M = W.mem[m];
                            const float4 mea = M.ea, meb = M.eb;
                            // (a member in act has this tile's array: its range is its own)
                            const uint32_t off = pos - M.lo, w = M.hi - M.lo;
                            const bool p0 = (off < w) & filter_box(r0, mea, meb);
                            const bool p1 = (off + 32 < w) & filter_box(r1, mea, meb);
                            const unsigned b0 = __ballot_sync(FULL, p0);
                            const unsigned b1 = __ballot_sync(FULL, p1);
                            if (!(b0 | b1)) continue;
                            if (p0)
                                W.plist[npl + __popc(b0 & lt_mask)] = (m << 8) | (uint32_t)lane;
                            if (p1)
                                W.plist[npl + __popc(b0) + __popc(b1 & lt_mask)] =
                                    (m << 8) | (uint32_t)(lane + 32);
                            npl += __popc(b0) + __popc(b1);
                        }
                        __syncwarp();
                        continue;
                    } else {
                        // stage 2: the bitmasks' survivors, one per lane per round, through the
                        // full box and gap filters
                        const bool have = (m0 | m1) != 0u;
                        const unsigned hv = __ballot_sync(FULL, have);
                        if (!hv) {
                            more = false;
                            break;
                        }
                        if (PASS == PASS_COUNT && lane == 0) W.count[3] += __popc(hv);
                        if (have) {
                            uint32_t i;
                            if (m0) {
                                i = __ffs(m0) - 1;
                                m0 &= m0 - 1u;
                            } else {
                                i = 31 + __ffs(m1);
                                m1 &= m1 - 1u;
                            }
                            const MemberRec &M = W.mem[lane];
                            const RecF r = C.r[i];
                            e = C.id[i];
                            qi = M.qi;
                            p = filter_box(r, M.ea, M.eb) &
                                filter_gap_e(r, M.ea, M.eb, W.ghdr.x, W.ghdr.y);
                        }
                    }
                    enqueue(p, qi, e);
                }
                if (qn >= 32) qn = pair_flush<PASS>(qn, false);
            }
            __syncwarp();
            if (pend) {
                if (lane == 0) copy_chunk(__ffs(pend) - 1, st);
                pend &= pend - 1u;
                pending |= 1u << st;
            }
        }
        if (abort) break;
        if (lane == 0) asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        t = __shfl_sync(FULL, t_next, 0);
        D = W.dnext;
        __syncwarp();  // (read by every lane before the next copy)
    }
    if (!abort && qn) pair_flush<PASS>(qn, true);
    // the unused slots of this warp's part hold no hit
    __syncwarp();
    if (PASS == PASS_COUNT)
        for (uint32_t j = W.sc_at + lane; j < W.sc_end; j += 32) B.s_tile[j] = 0xffffffffu;
    if (abort) {
        if (lane == 0) {
            atomicOr(B.status, DEV_ERR_TIMEOUT);
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
        // let copies still in flight land before the shared memory is released
        for (int st = 0; st < PK_STAGES; st++)
            if ((pending >> st) & 1u) mbar_wait_bounded(&W.bar[st], (parity >> st) & 1u);
        if (pending & MEM) mbar_wait_bounded(&W.mbar, (parity >> PK_STAGES) & 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0)
        atomicMax(&B.stats[PASS == PASS_COUNT ? ST_CNT1 : ST_WR1], (unsigned long long)globaltimer_ns());
    if (PASS == PASS_COUNT) {
        // the block's counts are summed in shared memory: one atomic per counter and block
        // (warps finish together, so per-warp atomics on these few addresses would queue)
        if (threadIdx.x < 6) {
            const WarpSmem *all = reinterpret_cast<const WarpSmem *>(smem_raw);
            unsigned long long v = 0;
            for (int w = 0; w < PK_WARPS; w++) v += all[w].count[threadIdx.x];
            const int slot = threadIdx.x < 4 ? ST_CHUNKS + (int)threadIdx.x
                                             : (threadIdx.x == 4 ? ST_EXACT : ST_HITS);
            if (v) atomicAdd(&B.stats[slot], v);
        }
    }
}

// Rows of the hits the count pass kept: row = the tile's scanned offset + the hit's rank in the
// tile, the same row the write pass's sweep would give it. When the scratch overflowed, the
// tiles it could not hold are swept again by the write pass (which writes the same values to the
// rows placed here). Does nothing when the rows exceed the output capacity.
__global__ void k_place(PipeBufs b, uint64_t scap, uint64_t tcap, uint64_t rows_cap)
{
    pdl_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0) b.stats[ST_WR0] = globaltimer_ns();
    const unsigned long long n = min((unsigned long long)scap, b.stats[ST_SCRATCH]);
    const uint64_t T = (uint64_t)b.hdr[HDR_T_LO] | ((uint64_t)b.hdr[HDR_T_HI] << 32);
    if (T > tcap || T > PK_MAX_TILES) return;  // overflow already flagged
    if (b.tile_off[T] > rows_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(b.status, DEV_ERR_OVERFLOW);
        return;
    }
    // four hits per thread at a time, their loads independent: a hit's tile offset waits for its
    // tile, and one such chain per thread left HBM idle (978 M hits, 56 B each at least: 23.3 ms
    // with one, 16.6 ms with four and a grid of several waves, 13.4 ms with a block's four
    // next to each other, 4.1 TB/s)
    for (uint64_t i0 = (uint64_t)blockIdx.x * 4 * TPB + threadIdx.x; i0 < n;
         i0 += (uint64_t)gridDim.x * 4 * TPB) {
        uint32_t t[4], rank[4], q[4], e[4];
        double tin[4], tout[4];
        uint64_t o[4], end[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint64_t i = i0 + k * TPB;
            t[k] = i < n ? __ldcs(b.s_tile + i) : 0xffffffffu;  // (a slot without a hit)
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint64_t i = i0 + k * TPB;
            const bool on = t[k] != 0xffffffffu;
            const uint32_t tk = on && t[k] < T ? t[k] : 0u;
            rank[k] = on ? __ldcs(b.s_rank + i) : 0u;
            q[k] = on ? __ldcs(b.s_q + i) : 0u;
            e[k] = on ? __ldcs(b.s_e + i) : 0u;
            tin[k] = on ? __ldcs(b.s_tin + i) : 0.0;
            tout[k] = on ? __ldcs(b.s_tout + i) : 0.0;
            o[k] = on ? b.tile_off[tk] : 0ull;
            end[k] = on ? b.tile_off[tk + 1] : 0ull;
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (t[k] == 0xffffffffu) continue;
            const uint64_t at = o[k] + rank[k];
            if (t[k] >= T || at >= end[k]) {
                atomicOr(b.status, DEV_ERR_INTERNAL);
                continue;
            }
            b.out_q[at] = q[k];
            b.out_e[at] = e[k];
            b.out_tin[at] = tin[k];
            b.out_tout[at] = tout[k];
        }
    }
}

constexpr size_t PAIR_SMEM = PK_WARPS * sizeof(WarpSmem) + sizeof(PairParams);
int g_pair_blocks = 0;

ts_status pair_grid(int *blocks)
{
    if (g_pair_blocks > 0) {
        *blocks = g_pair_blocks;
        return TS_OK;
    }
    int dev = 0, sms = 0, per = 0;
    TS_CUDA(cudaGetDevice(&dev));
    TS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int smem = (int)PAIR_SMEM;
    TS_CUDA(cudaFuncSetAttribute(k_pair<PASS_COUNT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    TS_CUDA(cudaFuncSetAttribute(k_pair<PASS_WRITE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    TS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<PASS_COUNT>, PK_THREADS, smem));
    if (per < 1) per = 1;
    g_pair_blocks = sms * per;
    *blocks = g_pair_blocks;
    return TS_OK;
}

void fill_pair_params(PairParams &P, const Index *ix, const PipeBufs &b, const PipeCaps &c)
{
    P.b = b;
    for (int k = 0; k < 3; k++) {
        P.rec[k] = ix->st_rec[k];
        P.box[k] = ix->st_box[k];
    }
    // ranges over the start-time order cover whole bins: they are swept in the copy in Morton
    // order inside every bin, chunk by chunk with the chunks' bounding records
    P.rec[SEL_T] = ix->trec;
    P.box[SEL_T] = ix->tbox;
    P.rec[SEL_GRID] = ix->ga_rec;
    P.box[SEL_GRID] = ix->gbox;
    P.seg = ix->seg;
    P.orig = ix->orig;
    P.tcap = c.tiles;
    P.rows_cap = c.rows;
    P.scap = c.scratch;
    P.exact_parts = c.exact_parts;
    P.tile = c.tile;
    P.tile_inv = (65536u + c.tile / PK_CH - 1) / (c.tile / PK_CH);
    P.stall_ns = 0;
}

// A stall requested for the next count pass (tests of the timeout path), taken by that launch.
std::atomic<uint64_t> g_stall_ns{0};

// Smallest float >= x (host).
float float_up(double x)
{
    float f = (float)x;
    if ((double)f < x) f = nextafterf(f, INFINITY);
    return f;
}

// Largest float <= x (host).
float float_dn(double x)
{
    float f = (float)x;
    if ((double)f > x) f = nextafterf(f, -INFINITY);
    return f;
}

int bits_for(uint64_t v)
{
    int b = 0;
    while (b < 64 && (v >> b) != 0) b++;
    return b;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// pipeline stages
// ---------------------------------------------------------------------------------------------
KeyFmt key_fmt(const Index *ix, const PipeCaps &c)
{
    const uint32_t nreq = c.nreq;
    uint64_t maxlen = ix->n;
    for (int d = 0; d < 3; d++) maxlen = std::max<uint64_t>(maxlen, ix->st_len[d]);
    maxlen = std::max<uint64_t>(maxlen, ix->g_len);
    KeyFmt f;
    f.sel_bits = ix->kind == TS_INDEX_SPATIOTEMPORAL ? 2 : 0;  // X, Y, Z or T
    const int full = bits_for(maxlen);  // bits of a range start
    const int head = 1 + f.sel_bits + bits_for(nreq > 1 ? nreq - 1 : 0);  // guard, array, request
    if (ix->kind == TS_INDEX_SPATIAL) {
        // as many start bits as keep the whole key within two 8-bit radix passes, but no fewer
        // than KEY_LO_MIN and no more than KEY_LO_BITS
        f.lo_bits = std::min(full, std::max(KEY_LO_MIN, std::min(KEY_LO_BITS, 16 - head)));
    } else {
        // three radix passes: as many of the start's top bits as tell the bins (or a subbin's bins)
        // apart, and the query's place; two passes where the pair kernel has too little to do for
        // the place to pay for the third (10,764 walk queries: it took 28 us either way)
        const int all = c.nq > 16384 ? 24 : 16;
        const int tell = bits_for(ix->m - 1) + 1 + (f.sel_bits ? 4 : 0);
        f.lo_bits = std::min(full, std::min(KEY_LO_BITS, std::max(1, std::min(tell, all - head))));
        if (all == 16 && nreq > 32) f.lo_bits = std::min(full, std::max(f.lo_bits, 8));
        f.morton = std::max(all == 16 ? 0 : 2, std::min(6, (all - head - f.lo_bits) / 3));
    }
    f.lo_shift = full - f.lo_bits;
    return f;
}

void fill_req(ReqDesc &r, const ts_query_params *qp, uint32_t q_first, uint32_t q_count)
{
    r.d = qp->d;
    r.dd = qp->d * qp->d;
    r.t_start = qp->t_start;
    r.t_end = qp->t_end;
    r.q_first = q_first;
    r.q_count = q_count;
    r.d_up = float_up(qp->d);
    r.d_dn = float_dn(qp->d);
    r.pad = 0.0f;
    for (int k = 0; k < 8; k++) r.cols[k] = nullptr;
    r.d2u = float_up(r.dd * (1.0 + 1e-6));
}

ts_status pipe_prepare(const Index *ix, const double *const cols[8], uint64_t nq,
                       const ReqDesc *reqs, uint32_t nreq, const PipeBufs &b, const PipeCaps &c,
                       cudaStream_t s)
{
    // cols == nullptr: every request's columns are read through its descriptor, and the run's
    // counters were reset by the caller
    if (cols) {
        TS_CUDA(cudaMemsetAsync(b.stats, 0, sizeof(unsigned long long) * ST_NSLOTS, s));
        TS_CUDA(cudaMemsetAsync(b.status, 0, sizeof(uint32_t), s));
        TS_CUDA(cudaMemsetAsync(b.counters, 0, sizeof(uint32_t) * 3, s));
        TS_CUDA(cudaMemsetAsync(b.req_units, 0, sizeof(uint32_t) * nreq, s));
    }
    PrepParams P;
    for (int k = 0; k < 8; k++) P.f[k] = cols ? cols[k] : nullptr;
    P.nq = nq;
    P.kind = ix->kind;
    P.reqs = reqs;
    P.nreq = nreq;
    P.kf = key_fmt(ix, c);
    P.mm = morton_map(ix, P.kf.morton);
    P.n = ix->n;
    P.m = ix->m;
    P.bin_start = ix->bin_start;
    P.bin_pmax = ix->bin_pmax;
    P.bin_off = ix->bin_off;
    P.bin_iwf = ix->b > 0.0 ? (float)(1.0 / ix->b) : 0.0f;
    {
        const double back = ix->b > 0.0 ? ceil(ix->max_dur / ix->b) + 2.0 : (double)ix->m;
        P.bin_back = back < (double)ix->m ? (uint32_t)back : ix->m;
    }
    for (int d = 0; d < 3; d++) {
        P.v[d] = ix->v[d];
        P.sub_bound[d] = ix->sub_bound[d];
        P.sub_iwf[d] = ix->sub_w[d] > 0.0 ? (float)(1.0 / ix->sub_w[d]) : 0.0f;
        P.st_off[d] = ix->st_off[d];
        P.g_bound[d] = ix->g_bound[d];
        P.g_iwf[d] = ix->g_w[d] > 0.0 ? (float)(1.0 / ix->g_w[d]) : 0.0f;
        P.longest[d] = ix->longest[d];
    }
    P.g = ix->g;
    P.b = b;
    // lookup tables in shared memory when they fit
    uint64_t tb = 0;
    if (ix->kind == TS_INDEX_SPATIAL) {
        tb = 3ull * 8 * ((uint64_t)ix->g + 1);
    } else if (ix->kind != TS_INDEX_BRUTE) {
        tb = 16ull * ix->m + 4ull * ((uint64_t)ix->m + 1);
        if (ix->kind == TS_INDEX_SPATIOTEMPORAL)
            for (int d = 0; d < 3; d++) tb += 8ull * ((uint64_t)ix->v[d] + 1);
    }
    P.smem_bytes = tb <= QP_TABLE_BYTES ? (uint32_t)tb : 0u;
    if (nq) {
        TS_LAUNCH_PDL(k_qprep, dim3(nblk(nq)), dim3(TPB), P.smem_bytes, s,
                      P);
    }
    return TS_OK;
}

ts_status pipe_grid_units(const Index *ix, uint64_t nq, const PipeBufs &b, const PipeCaps &c,
                          cudaStream_t s, bool all_or_none)
{
    if (!nq) return TS_OK;
    const unsigned ublk = (unsigned)std::min<uint64_t>((nq + TPB - 1) / TPB, 152 * 16);
    TS_LAUNCH_PDL(k_grid_units, dim3(ublk), dim3(TPB), 0, s,
                  nq, c.units, key_fmt(ix, c), ix->g, ix->g_off, all_or_none, b);
    return TS_OK;
}

ts_status pipe_group(const Index *ix, const ReqDesc *reqs, uint32_t nreq, const PipeBufs &b,
                     const PipeCaps &c, bool host_tiles,
                     cudaStream_t s)
{
    // one bit above the key fields: a unit without candidates has key ~0 and sorts last
    const KeyFmt f = key_fmt(ix, c);
    const int bits =
        3 * f.morton + f.lo_bits + f.sel_bits + bits_for(c.nreq > 1 ? c.nreq - 1 : 0) + 1;
    TS_CHECK(radix_sort_u64(b.keys, b.vals, c.units, bits, s, b.hdr + HDR_NU, false));
    if (nreq > 1) {
        TS_LAUNCH_PDL(k_req_scan, dim3(1), dim3(32), 0, s,
                      nreq, b);
    }
    const unsigned gblk = (unsigned)std::min<uint64_t>((c.groups * 32 + TPB - 1) / TPB, 152 * 16);
    TS_LAUNCH_PDL(k_groups, dim3(gblk), dim3(TPB), 0, s,
                  nreq, c.groups, c.tile, reqs, b);
    TS_CHECK(scan_u32_to_u64(b.ntiles, b.tile_base, c.groups, s, b.hdr + HDR_G));
    if (host_tiles) {  // the caller reads the tile count before the count pass
        TS_LAUNCH_PDL(k_hdr, dim3(1), dim3(1), 0, s,
                      c.groups, c.tiles, b);
    }
    return TS_OK;
}

ts_status pair_warps(const PipeCaps &c, uint64_t *warps)
{
    int blocks = 0;
    TS_CHECK(pair_grid(&blocks));
    if (c.pair_blocks > 0 && c.pair_blocks < blocks) blocks = c.pair_blocks;
    *warps = (uint64_t)blocks * PK_WARPS;
    return TS_OK;
}

ts_status pipe_count(const Index *ix, const PipeBufs &b, const PipeCaps &c,
                     cudaStream_t s)
{
    int blocks = 0;
    TS_CHECK(pair_grid(&blocks));
    if (c.pair_blocks > 0 && c.pair_blocks < blocks) blocks = c.pair_blocks;
    PairParams P;
    fill_pair_params(P, ix, b, c);
    P.stall_ns = c.stall_ns;
    if (c.tiles) {
        ArrayPtrs<const RecF> box;
        for (int k = 0; k < 5; k++) box.p[k] = P.box[k];
        const unsigned dblk = (unsigned)std::min<uint64_t>(
            std::max<uint64_t>((c.groups * 32 + TPB - 1) / TPB, (c.tiles + TPB - 1) / TPB), 152 * 8);
        TS_LAUNCH_PDL(k_tile_desc, dim3(dblk), dim3(TPB), 0, s,
                      c.groups, c.tiles, c.tile, (uint32_t)(blocks * PK_WARPS), box, b);
        TS_LAUNCH_PDL(k_pair<PASS_COUNT>, dim3(blocks), dim3(PK_THREADS),
                      PAIR_SMEM, s, P);
    }
    return TS_OK;
}

void inject_stall(uint64_t ns) { g_stall_ns.store(ns); }

ts_status pipe_scan_rows(const PipeBufs &b, const PipeCaps &c, cudaStream_t s)
{
    return scan_u32_to_u64(b.tile_hits, b.tile_off, c.tiles, s, b.hdr + HDR_T_LO, ~TILE_REDO);
}

ts_status pipe_write(const Index *ix, const PipeBufs &b, const PipeCaps &c, cudaStream_t s)
{
    int blocks = 0;
    TS_CHECK(pair_grid(&blocks));
    if (c.pair_blocks > 0 && c.pair_blocks < blocks) blocks = c.pair_blocks;
    PairParams P;
    fill_pair_params(P, ix, b, c);
    if (c.tiles) {
        TS_LAUNCH_PDL(k_place, dim3(152 * 32), dim3(TPB), 0, s,
                      b, c.scratch, c.tiles, c.rows);
        TS_LAUNCH_PDL(k_pair<PASS_WRITE>, dim3(blocks), dim3(PK_THREADS),
                      PAIR_SMEM, s, P);
    }
    return TS_OK;
}

// ---------------------------------------------------------------------------------------------
// host orchestration of one plain search
// ---------------------------------------------------------------------------------------------
ts_status read_dev_status(uint32_t st)
{
    if (st & DEV_ERR_INVALID) {
        set_error("invalid query segment (NaN/Inf or t_end <= t_start)");
        return TS_ERR_INVALID_ARG;
    }
    if (st & DEV_ERR_TIMEOUT) {
        set_error("a bounded device wait ran out (bulk copy did not complete)");
        return TS_ERR_TIMEOUT;
    }
    if (st & DEV_ERR_OVERFLOW) {
        set_error("a work buffer capacity was exceeded");
        return TS_ERR_CAPACITY;
    }
    if (st) {
        set_error("search: device status 0x%x", st);
        return TS_ERR_INTERNAL;
    }
    return TS_OK;
}

ts_status device_cols(const ts_segments *q, cudaStream_t s, DevBuf &copy, const double *cols[8])
{
    const double *src[8] = {q->x0, q->y0, q->z0, q->t0, q->x1, q->y1, q->z1, q->t1};
    for (int k = 0; k < 8; k++)
        if (!src[k] && q->n) {
            set_error("NULL query column %d", k);
            return TS_ERR_INVALID_ARG;
        }
    if (!q->on_host) {
        for (int k = 0; k < 8; k++) cols[k] = src[k];
        return TS_OK;
    }
    TS_CHECK(copy.alloc(sizeof(double) * q->n * 8, s));
    for (int k = 0; k < 8; k++) {
        double *dst = copy.as<double>() + (uint64_t)k * q->n;
        TS_CUDA(cudaMemcpyAsync(dst, src[k], sizeof(double) * q->n, cudaMemcpyHostToDevice, s));
        cols[k] = dst;
    }
    return TS_OK;
}

ts_status check_query_params(const ts_query_params *qp)
{
    if (!qp) {
        set_error("NULL query parameters");
        return TS_ERR_INVALID_ARG;
    }
    if (!(qp->d > 0.0) || !isfinite(qp->d)) {
        set_error("d must be finite and > 0 (got %g)", qp->d);
        return TS_ERR_INVALID_ARG;
    }
    if (isnan(qp->t_start) || isnan(qp->t_end) || qp->t_start > qp->t_end) {
        set_error("query interval must satisfy t_start <= t_end");
        return TS_ERR_INVALID_ARG;
    }
    return TS_OK;
}

namespace {

// Work buffers of a plain search, allocated stage by stage at their exact sizes.
struct PlainWork {
    DevBuf qd, qf, qreq, qcell, qnu, quoff, u_q, u_lo, u_hi, u_sel, keys, vals, req, groups, segs,
        ntiles, tile_base, tiles, tdesc, tile_off, ctl, reqdesc, scratch, gmem;
};

ts_status alloc_units(PlainWork &w, PipeBufs &b, uint64_t units, cudaStream_t s)
{
    TS_CHECK(w.u_q.alloc(sizeof(uint32_t) * units, s));
    TS_CHECK(w.u_lo.alloc(sizeof(uint32_t) * units, s));
    TS_CHECK(w.u_hi.alloc(sizeof(uint32_t) * units, s));
    TS_CHECK(w.u_sel.alloc(sizeof(uint32_t) * units, s));
    TS_CHECK(w.keys.alloc(sizeof(uint64_t) * units, s));
    TS_CHECK(w.vals.alloc(sizeof(uint32_t) * units, s));
    b.u_q = w.u_q.as<uint32_t>();
    b.u_lo = w.u_lo.as<uint32_t>();
    b.u_hi = w.u_hi.as<uint32_t>();
    b.u_sel = w.u_sel.as<uint32_t>();
    b.keys = w.keys.as<uint64_t>();
    b.vals = w.vals.as<uint32_t>();
    return TS_OK;
}

ts_status plain_prepare(const Index *ix, const double *const cols[8], uint64_t nq,
                        const ts_query_params *qp, cudaStream_t s, PlainWork &w, PipeBufs &b,
                        PipeCaps &c, bool group)
{
    b = PipeBufs{};
    c = PipeCaps{};
    c.nq = nq;
    c.nreq = 1;
    ReqDesc rd;
    fill_req(rd, qp, 0, (uint32_t)nq);
    TS_CHECK(w.reqdesc.alloc(sizeof(ReqDesc), s));
    TS_CUDA(cudaMemcpyAsync(w.reqdesc.p, &rd, sizeof(ReqDesc), cudaMemcpyHostToDevice, s));
    TS_CHECK(w.qd.alloc(sizeof(QueryD) * nq, s));
    TS_CHECK(w.qf.alloc(sizeof(float4) * 2 * nq, s));
    TS_CHECK(w.qreq.alloc(sizeof(uint32_t) * nq, s));
    // control block: hdr (8 u32), stats (ST_NSLOTS u64), status, 3 counters
    TS_CHECK(w.ctl.alloc(256, s));
    TS_CHECK(w.req.alloc(sizeof(uint32_t) * 8, s));
    b.qd = w.qd.as<QueryD>();
    b.qf = w.qf.as<float4>();
    b.qreq = w.qreq.as<uint32_t>();
    b.hdr = w.ctl.as<uint32_t>();
    b.stats = reinterpret_cast<unsigned long long *>(w.ctl.as<uint32_t>() + 8);
    b.status = w.ctl.as<uint32_t>() + 8 + 2 * ST_NSLOTS;
    b.counters = b.status + 1;
    b.req_units = w.req.as<uint32_t>();
    b.ustart = b.req_units + 1;
    b.req_groups = b.req_units + 3;
    b.gstart = b.req_units + 4;
    uint64_t units = nq;
    if (ix->kind == TS_INDEX_SPATIAL) {
        TS_CHECK(w.qcell.alloc(sizeof(uint32_t) * 2 * nq, s));
        TS_CHECK(w.qnu.alloc(sizeof(uint32_t) * nq, s));
        TS_CHECK(w.quoff.alloc(sizeof(uint32_t) * (nq + 1), s));
        b.qcell = w.qcell.as<uint32_t>();
        b.qnu = w.qnu.as<uint32_t>();
        b.quoff = w.quoff.as<uint32_t>();
    } else {
        TS_CHECK(alloc_units(w, b, nq, s));
    }
    TS_CHECK(pipe_prepare(ix, cols, nq, w.reqdesc.as<ReqDesc>(), 1, b, c, s));
    if (ix->kind == TS_INDEX_SPATIAL) {
        TS_CHECK(scan_u32(b.qnu, b.quoff, nq, b.status, s));
        uint32_t total = 0;
        TS_CUDA(cudaMemcpyAsync(&total, b.quoff + nq, 4, cudaMemcpyDeviceToHost, s));
        TS_CUDA(cudaStreamSynchronize(s));
        units = total;
        TS_CHECK(alloc_units(w, b, units, s));
        c.units = units;
        TS_CHECK(pipe_grid_units(ix, nq, b, c, s));
    }
    c.units = units;
    if (!group) return TS_OK;
    c.groups = (units + GROUP - 1) / GROUP + 1;
    TS_CHECK(w.groups.alloc(sizeof(uint32_t) * c.groups, s));
    TS_CHECK(w.gmem.alloc((sizeof(MemberRec) * GROUP + 3 * sizeof(float4)) * c.groups, s));
    b.gmem = w.gmem.as<MemberRec>();
    b.ghdr = reinterpret_cast<float4 *>(b.gmem + GROUP * c.groups);
    TS_CHECK(w.segs.alloc(sizeof(uint32_t) * 4 * GROUP * c.groups, s));
    TS_CHECK(w.ntiles.alloc(sizeof(uint32_t) * c.groups, s));
    TS_CHECK(w.tile_base.alloc(sizeof(uint64_t) * (c.groups + 1), s));
    b.g_nseg = w.groups.as<uint32_t>();
    b.seg_lo = w.segs.as<uint32_t>();
    b.seg_hi = b.seg_lo + GROUP * c.groups;
    b.seg_sel = b.seg_hi + GROUP * c.groups;
    b.seg_t0 = b.seg_sel + GROUP * c.groups;
    b.ntiles = w.ntiles.as<uint32_t>();
    b.tile_base = w.tile_base.as<uint64_t>();
    c.tiles = ~0ull;  // sized after the grouping; no overflow check in the header kernel
    TS_CHECK(pipe_group(ix, w.reqdesc.as<ReqDesc>(), 1, b, c, true, s));
    return TS_OK;
}

void fill_stats(const unsigned long long *h, ts_search_stats *st);

ts_status copy_stats(const PipeBufs &b, cudaStream_t s, ts_search_stats *st, uint32_t *status)
{
    unsigned long long h[ST_NSLOTS];
    TS_CUDA(cudaMemcpyAsync(h, b.stats, sizeof(h), cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(status, b.status, 4, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    fill_stats(h, st);
    return TS_OK;
}

void fill_stats(const unsigned long long *h, ts_search_stats *st)
{
    st->n_qsegs = h[ST_QSEGS];
    st->n_tests = h[ST_TESTS];
    st->n_exact = h[ST_EXACT];
    st->n_hits = h[ST_HITS];
    st->n_tiles = h[ST_TILES];
    st->n_groups = h[ST_GROUPS];
    st->n_subbin = h[ST_SUBBIN];
    st->n_chunks = h[ST_CHUNKS];
    st->n_dense = h[ST_DENSE];
    st->n_sparse = h[ST_SPARSE];
    st->n_stage2 = h[ST_STAGE2];
    st->ms_count_pass = stamp_ms(h[ST_CNT0], h[ST_CNT1]);
    st->ms_write_pass = stamp_ms(h[ST_WR0], h[ST_WR1]);
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// a search in one go: every kernel enqueued at once on guessed capacities, one wait
// ---------------------------------------------------------------------------------------------
namespace {

constexpr uint64_t ONE_GO_QUERIES = 1ull << 16;  // above, the kernels dwarf the waits
constexpr uint64_t ONE_GO_ROWS = 1ull << 16;     // rows a result may have room for unasked
constexpr uint64_t ONE_GO_UNITS = 1ull << 22;    // (3 KB of work buffers each 32)
constexpr uint64_t ONE_GO_TILES = 1ull << 24;    // (28 B of work buffers each)
constexpr uint64_t STAGE_QUERIES = 1024;         // host queries read in place from pinned memory

// Runs of cells of a query no longer than the longest entry: its extents in x and y, d more on
// both sides and the longest entry's more below, in cells. (A first guess of 16 was too small for
// d of several cells, and a dense search on the grid ran twice: 403 -> 503 us.)
uint64_t grid_runs(const Index *ix, double d)
{
    uint64_t runs = 1;
    for (int k = 0; k < 2; k++) {
        const double cells = ix->g_w[k] > 0.0 ? ceil((2.0 * d + 2.0 * ix->longest[k]) / ix->g_w[k]) + 1.0
                                              : 1.0;
        runs *= cells < (double)ix->g ? (uint64_t)cells : (uint64_t)ix->g;
    }
    return runs;
}

// About the most tiles of a group: all entries without bins, with bins those of the bins that a query
// of this window (negative: as long as the longest entry's) meets and a few more; a few runs of
// cells on the grid.
uint64_t group_tiles(const Index *ix, double window)
{
    if (ix->kind == TS_INDEX_SPATIAL) return 64;
    double n = (double)ix->n;
    if (ix->kind != TS_INDEX_BRUTE && ix->b > 0.0)
        n = std::min(n, (ceil((window < 0.0 ? ix->max_dur : window) / ix->b) +
                         ceil(ix->max_dur / ix->b) + 8.0) * (n / ix->m));
    return (uint64_t)(n / PK_TILE) + GROUP + 2;
}

// What the host reads after the wait.
struct PlainOut {
    uint32_t hdr[8];
    unsigned long long stats[ST_NSLOTS];
    unsigned long long total;
    uint32_t status, units;
};

// Pinned, mapped memory of one search in flight: its outcome and its small host query set.
struct HostSlot {
    PlainOut out;
    alignas(256) double stage[8 * STAGE_QUERIES];
};

// A fixed number of slots for the searches in flight, allocated once; a search that finds none
// free takes the stepwise path.
class SlotPool {
public:
    HostSlot *take()
    {
        std::lock_guard<std::mutex> lk(mu_);
        if (!base_ && !failed_) {
            void *p = nullptr;
            if (cudaHostAlloc(&p, sizeof(HostSlot) * SLOTS,
                              cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) {
                base_ = static_cast<HostSlot *>(p);
            } else {
                cudaGetLastError();
                failed_ = true;
            }
        }
        for (int k = 0; base_ && k < SLOTS; k++)
            if (!((used_ >> k) & 1u)) {
                used_ |= 1u << k;
                return base_ + k;
            }
        return nullptr;
    }
    void give(HostSlot *h)
    {
        std::lock_guard<std::mutex> lk(mu_);
        used_ &= ~(1u << (h - base_));
    }

private:
    static constexpr int SLOTS = 16;
    std::mutex mu_;
    HostSlot *base_ = nullptr;
    uint32_t used_ = 0;
    bool failed_ = false;
};
SlotPool g_slots;

__global__ void k_plain_start(ReqDesc rd, ReqDesc *reqs, PipeBufs b)
{
    pdl_enter();
    const uint32_t t = threadIdx.x;
    if (t < 8) b.hdr[t] = 0;
    if (t < ST_NSLOTS) b.stats[t] = 0;
    if (t < 3) b.counters[t] = 0;
    if (t == 0) {
        *b.status = 0;
        b.req_units[0] = 0;
        *reqs = rd;
    }
}

__global__ void k_plain_out(uint64_t nq, uint64_t tcap, PipeBufs b, PlainOut *out)
{
    pdl_enter();
    const uint32_t t = threadIdx.x;
    const uint64_t T = (uint64_t)b.hdr[HDR_T_LO] | ((uint64_t)b.hdr[HDR_T_HI] << 32);
    if (t < 8) out->hdr[t] = b.hdr[t];
    if (t < ST_NSLOTS) out->stats[t] = b.stats[t];
    if (t == 0) {
        out->total = T <= tcap ? b.tile_off[T] : 0ull;
        out->status = *b.status;
        out->units = b.quoff ? b.quoff[nq] : 0u;
    }
}

void plain_layout(Carver &k, const PipeCaps &c, bool grid, PipeBufs &b, ReqDesc **reqs)
{
    *reqs = k.take<ReqDesc>(1);
    b.hdr = k.take<uint32_t>(8);
    b.stats = k.take<unsigned long long>(ST_NSLOTS);
    b.status = k.take<uint32_t>(4);
    b.counters = b.status + 1;
    b.req_units = k.take<uint32_t>(8);
    b.ustart = b.req_units + 1;
    b.req_groups = b.req_units + 3;
    b.gstart = b.req_units + 4;
    b.qd = k.take<QueryD>(c.nq);
    b.qf = k.take<float4>(2 * c.nq);
    b.qreq = k.take<uint32_t>(c.nq);
    b.qcell = grid ? k.take<uint32_t>(2 * c.nq) : nullptr;
    b.qnu = grid ? k.take<uint32_t>(c.nq) : nullptr;
    b.quoff = grid ? k.take<uint32_t>(c.nq + 1) : nullptr;
    b.u_q = k.take<uint32_t>(c.units);
    b.u_lo = k.take<uint32_t>(c.units);
    b.u_hi = k.take<uint32_t>(c.units);
    b.u_sel = k.take<uint32_t>(c.units);
    b.keys = k.take<uint64_t>(c.units);
    b.vals = k.take<uint32_t>(c.units);
    b.g_nseg = k.take<uint32_t>(c.groups);
    b.gmem = k.take<MemberRec>(GROUP * c.groups);
    b.ghdr = k.take<float4>(3 * c.groups);
    b.seg_lo = k.take<uint32_t>(GROUP * c.groups);
    b.seg_hi = k.take<uint32_t>(GROUP * c.groups);
    b.seg_sel = k.take<uint32_t>(GROUP * c.groups);
    b.seg_t0 = k.take<uint32_t>(GROUP * c.groups);
    b.ntiles = k.take<uint32_t>(c.groups);
    b.tile_base = k.take<uint64_t>(c.groups + 1);
    b.tdesc = k.take<uint4>(c.tiles);
    b.tile_hits = k.take<uint32_t>(c.tiles);
    b.tile_off = k.take<uint64_t>(c.tiles + 1);
    b.s_tile = k.take<uint32_t>(c.scratch);
    b.s_rank = k.take<uint32_t>(c.scratch);
    b.s_q = k.take<uint32_t>(c.scratch);
    b.s_e = k.take<uint32_t>(c.scratch);
    b.s_tin = k.take<double>(c.scratch);
    b.s_tout = k.take<double>(c.scratch);
}

void free_rows(SearchOut *out, cudaStream_t s)
{
    for (void *p : {(void *)out->q, (void *)out->e, (void *)out->tin, (void *)out->tout})
        if (p) cudaFreeAsync(p, s);
    out->q = out->e = nullptr;
    out->tin = out->tout = nullptr;
}

ts_status alloc_rows(SearchOut *out, uint64_t n, cudaStream_t s, PipeBufs &b)
{
    TS_CUDA(pool_malloc((void **)&out->q, sizeof(uint32_t) * n, s));
    TS_CUDA(pool_malloc((void **)&out->e, sizeof(uint32_t) * n, s));
    TS_CUDA(pool_malloc((void **)&out->tin, sizeof(double) * n, s));
    TS_CUDA(pool_malloc((void **)&out->tout, sizeof(double) * n, s));
    b.out_q = out->q;
    b.out_e = out->e;
    b.out_tin = out->tin;
    b.out_tout = out->tout;
    return TS_OK;
}

// The search with work buffers of guessed sizes in one allocation, every kernel enqueued before
// the one wait. *done stays false, and nothing is kept, when a guess was too small, memory or a
// slot was short: the stepwise path below, which waits for every size, then answers (also with
// its errors). Up to ONE_GO_ROWS rows (8 per query) are in place after the wait; more take their
// exact arrays and a second one.
//
// Bound: launches and their latency. A search of 20 query segments against 20,000 (34 calls to the
// allocator, 12 pageable copies, four waits, 18 kernels before) 327 -> 207 us, of 10,000
// against 1M on the grid 395 -> 245 us, with the binding and the copies of the rows.
ts_status one_go_steps(const Index *ix, const ts_segments *q, const ts_query_params *qp,
                       double window, cudaStream_t s, SearchOut *out, bool *done)
{
    const uint64_t nq = q->n;
    const bool grid = ix->kind == TS_INDEX_SPATIAL;
    struct Slot {
        HostSlot *h = g_slots.take();
        cudaStream_t busy = nullptr;
        bool is_busy = false;  // kernels that use the slot may be in flight (an error in between)
        ~Slot()
        {
            if (is_busy) cudaStreamSynchronize(busy);
            if (h) g_slots.give(h);
        }
    } slot;
    if (!slot.h) return TS_OK;
    PlainOut *dout = nullptr;
    {
        void *p = nullptr;
        if (cudaHostGetDevicePointer(&p, slot.h, 0) != cudaSuccess) {
            cudaGetLastError();
            return TS_OK;
        }
        dout = static_cast<PlainOut *>(p);
    }
    PipeCaps c;
    c.nq = nq;
    c.nreq = 1;
    c.units = grid ? nq * grid_runs(ix, qp->d) + 1024 : nq;
    c.groups = c.units / GROUP + 2;
    c.tiles = group_tiles(ix, window) * c.groups + 65536;
    if (c.units > ONE_GO_UNITS || c.tiles > ONE_GO_TILES) return TS_OK;
    uint64_t warps = 0;
    TS_CHECK(pair_warps(c, &warps));
    c.scratch = scratch_slots(std::min<uint64_t>(std::max<uint64_t>(4 * nq + (1ull << 20), 512 * nq),
                                                 SCRATCH_MAX), warps);
    c.rows = std::min<uint64_t>(8 * nq + 64, ONE_GO_ROWS);
    PipeBufs b = PipeBufs{};
    ReqDesc *reqs = nullptr;
    Carver size;
    plain_layout(size, c, grid, b, &reqs);
    DevBuf arena;
    if (arena.alloc(size.off, s) != TS_OK) return TS_OK;
    Carver cut;
    cut.base = arena.as<unsigned char>();
    plain_layout(cut, c, grid, b, &reqs);

    const double *src[8] = {q->x0, q->y0, q->z0, q->t0, q->x1, q->y1, q->z1, q->t1};
    DevBuf qcopy;
    const double *cols[8];
    if (q->on_host && nq <= STAGE_QUERIES) {
        for (int k = 0; k < 8; k++) {
            if (!src[k]) return TS_OK;  // (the stepwise path names the column)
            memcpy(slot.h->stage + k * nq, src[k], sizeof(double) * nq);
            cols[k] = reinterpret_cast<const double *>(reinterpret_cast<unsigned char *>(dout) +
                                                       offsetof(HostSlot, stage)) + k * nq;
        }
    } else {
        *done = true;
        TS_CHECK(device_cols(q, s, qcopy, cols));
        *done = false;
    }
    ReqDesc rd;
    fill_req(rd, qp, 0, (uint32_t)nq);
    for (int k = 0; k < 8; k++) rd.cols[k] = cols[k];
    *done = true;  // (every return below but those that say otherwise)
    TS_CHECK(alloc_rows(out, c.rows, s, b));
    slot.busy = s;
    slot.is_busy = true;
    TS_LAUNCH_PDL(k_plain_start, dim3(1), dim3(32), 0, s, rd, reqs, b);
    TS_CHECK(pipe_prepare(ix, nullptr, nq, reqs, 1, b, c, s));
    if (grid) {
        TS_CHECK(scan_u32(b.qnu, b.quoff, nq, b.status, s));
        TS_CHECK(pipe_grid_units(ix, nq, b, c, s, true));
    }
    TS_CHECK(pipe_group(ix, reqs, 1, b, c, false, s));
    c.stall_ns = g_stall_ns.exchange(0);  // (a stall requested by a test of the timeout path)
    TS_CHECK(pipe_count(ix, b, c, s));
    TS_CHECK(pipe_scan_rows(b, c, s));
    TS_CHECK(pipe_write(ix, b, c, s));
    TS_LAUNCH_PDL(k_plain_out, dim3(1), dim3(32), 0, s, nq, c.tiles, b, dout);
    TS_CUDA(cudaStreamSynchronize(s));
    slot.is_busy = false;
    const PlainOut &o = slot.h->out;
    TS_CHECK(read_dev_status(o.status & ~(uint32_t)DEV_ERR_OVERFLOW));
    const uint64_t T = (uint64_t)o.hdr[HDR_T_LO] | ((uint64_t)o.hdr[HDR_T_HI] << 32);
    if (o.units > c.units || T > c.tiles) {  // a guess was too small
        free_rows(out, s);
        *done = false;
        return TS_OK;
    }
    fill_stats(o.stats, &out->stats);
    out->stats.n_queries = nq;
    const uint64_t total = o.total;
    out->count = total;
    if (out->stats.n_hits != total) {
        set_error("hit count mismatch (%llu vs %llu)", (unsigned long long)out->stats.n_hits,
                  (unsigned long long)total);
        return TS_ERR_INTERNAL;
    }
    if (total == 0 || total > c.rows) free_rows(out, s);
    if (qp->max_results && total > qp->max_results) {
        free_rows(out, s);
        set_error("%llu result rows exceed max_results %llu", (unsigned long long)total,
                  (unsigned long long)qp->max_results);
        return TS_ERR_CAPACITY;
    }
    if (total <= c.rows) return TS_OK;
    TS_CHECK(alloc_rows(out, total, s, b));
    c.rows = total;
    c.stall_ns = 0;
    slot.is_busy = true;
    TS_CUDA(cudaMemsetAsync(b.status, 0, sizeof(uint32_t), s));  // (the rows' overflow)
    TS_CHECK(pipe_write(ix, b, c, s));
    TS_LAUNCH_PDL(k_plain_out, dim3(1), dim3(32), 0, s, nq, c.tiles, b, dout);
    TS_CUDA(cudaStreamSynchronize(s));
    slot.is_busy = false;
    TS_CHECK(read_dev_status(o.status));
    fill_stats(o.stats, &out->stats);
    out->stats.n_queries = nq;
    return TS_OK;
}

// (memory may also run short after the arena: for the query copy, a sort's or a scan's buffers, the
// rows. What was enqueued has ended by then, and the arena is back in the pool.)
ts_status search_one_go(const Index *ix, const ts_segments *q, const ts_query_params *qp,
                        double window, cudaStream_t s, SearchOut *out, bool *done)
{
    const ts_status st = one_go_steps(ix, q, qp, window, s, out, done);
    if (st != TS_ERR_OOM) return st;
    free_rows(out, s);
    out->count = 0;
    out->stats = ts_search_stats{};
    out->stats.n_queries = q->n;
    *done = false;
    return TS_OK;
}

}  // namespace

ts_status search_plain(const Index *ix, const ts_segments *q, const ts_query_params *qp,
                       cudaStream_t s, SearchOut *out, double window)
{
    TS_CHECK(check_query_params(qp));
    if (!q) {
        set_error("NULL query set");
        return TS_ERR_INVALID_ARG;
    }
    if (q->n > 0x7fffffffull) {
        set_error("query set larger than 2^31 - 1 segments");
        return TS_ERR_INVALID_ARG;
    }
    *out = SearchOut{};
    const uint64_t nq = q->n;
    out->stats.n_queries = nq;
    out->n_entries = ix->n;
    if (nq == 0) return TS_OK;
    if (nq <= ONE_GO_QUERIES) {
        bool done = false;
        const ts_status got = search_one_go(ix, q, qp, window, s, out, &done);
        if (done) return got;
    }
    DevBuf qcopy;
    const double *cols[8];
    TS_CHECK(device_cols(q, s, qcopy, cols));
    PlainWork w;
    PipeBufs b;
    PipeCaps c;
    TS_CHECK(plain_prepare(ix, cols, nq, qp, s, w, b, c, true));

    uint32_t hdr[HDR_N];
    uint32_t st = 0;
    TS_CUDA(cudaMemcpyAsync(hdr, b.hdr, sizeof(hdr), cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(&st, b.status, 4, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    TS_CHECK(read_dev_status(st));
    c.tiles = (uint64_t)hdr[HDR_T_LO] | ((uint64_t)hdr[HDR_T_HI] << 32);
    TS_CHECK(w.tiles.alloc(sizeof(uint32_t) * (c.tiles ? c.tiles : 1), s));
    TS_CHECK(w.tdesc.alloc(sizeof(uint4) * (c.tiles ? c.tiles : 1), s));
    TS_CHECK(w.tile_off.alloc(sizeof(uint64_t) * (c.tiles + 1), s));
    b.tdesc = w.tdesc.as<uint4>();
    b.tile_hits = w.tiles.as<uint32_t>();
    // hits kept by the count pass and placed after the scan (a second sweep when they overflow)
    uint64_t warps = 0;
    TS_CHECK(pair_warps(c, &warps));
    c.scratch = scratch_slots(std::min<uint64_t>(std::max<uint64_t>(4 * nq + (1ull << 20), 512 * nq),
                                                 SCRATCH_MAX), warps);
    if (w.scratch.alloc(32 * c.scratch, s) != TS_OK) {  // (short of memory: sweep twice instead)
        c.scratch = std::min<uint64_t>(4 * nq + (1ull << 20), SCRATCH_MAX);
        TS_CHECK(w.scratch.alloc(32 * c.scratch, s));
    }
    b.s_tile = w.scratch.as<uint32_t>();
    b.s_rank = b.s_tile + c.scratch;
    b.s_q = b.s_rank + c.scratch;
    b.s_e = b.s_q + c.scratch;
    b.s_tin = reinterpret_cast<double *>(b.s_e + c.scratch);
    b.s_tout = b.s_tin + c.scratch;
    b.tile_off = w.tile_off.as<uint64_t>();

    c.stall_ns = g_stall_ns.exchange(0);  // (a stall requested by a test of the timeout path)
    TS_CHECK(pipe_count(ix, b, c, s));
    TS_CHECK(pipe_scan_rows(b, c, s));
    uint64_t total = 0;
    TS_CUDA(cudaMemcpyAsync(&total, b.tile_off + c.tiles, 8, cudaMemcpyDeviceToHost, s));
    TS_CHECK(copy_stats(b, s, &out->stats, &st));
    TS_CHECK(read_dev_status(st));
    out->stats.n_queries = nq;
    out->count = total;
    if (out->stats.n_hits != total) {
        set_error("hit count mismatch (%llu vs %llu)", (unsigned long long)out->stats.n_hits,
                  (unsigned long long)total);
        return TS_ERR_INTERNAL;
    }
    if (qp->max_results && total > qp->max_results) {
        set_error("%llu result rows exceed max_results %llu", (unsigned long long)total,
                  (unsigned long long)qp->max_results);
        return TS_ERR_CAPACITY;
    }
    if (total == 0) return TS_OK;
    TS_CUDA(pool_malloc((void **)&out->q, sizeof(uint32_t) * total, s));
    TS_CUDA(pool_malloc((void **)&out->e, sizeof(uint32_t) * total, s));
    TS_CUDA(pool_malloc((void **)&out->tin, sizeof(double) * total, s));
    TS_CUDA(pool_malloc((void **)&out->tout, sizeof(double) * total, s));
    b.out_q = out->q;
    b.out_e = out->e;
    b.out_tin = out->tin;
    b.out_tout = out->tout;
    c.rows = total;
    TS_CHECK(pipe_write(ix, b, c, s));
    TS_CHECK(copy_stats(b, s, &out->stats, &st));
    return read_dev_status(st);
}

// Rows, in their order or in `order`, into one block of memory (a slot's pinned one, or the device's):
// t_in, t_out, q_idx, e_idx.
__global__ void k_rows_out(uint64_t n, const uint32_t *order, const uint32_t *q, const uint32_t *e,
                           const double *tin, const double *tout, double *to)
{
    pdl_enter();
    uint32_t *w = reinterpret_cast<uint32_t *>(to + 2 * n);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t r = order ? order[i] : i;
        to[i] = tin[r];
        to[n + i] = tout[r];
        w[i] = q[r];
        w[n + i] = e[r];
    }
}

__global__ void k_row_keys(uint64_t n, const uint32_t *q, const uint32_t *e, int ebits,
                           uint64_t *keys, uint32_t *vals)
{
    pdl_enter();
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        keys[i] = ((uint64_t)q[i] << ebits) | e[i];
        vals[i] = (uint32_t)i;
    }
}

// Whether kernels of the current device may read the rows.
bool rows_here(const SearchOut &o)
{
    int dev = -1;
    cudaPointerAttributes pa;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaPointerGetAttributes(&pa, o.q) == cudaSuccess &&
        pa.device == dev)
        return true;
    cudaGetLastError();
    return false;
}

// Few rows reach pageable host memory through a slot, in one kernel and one wait (four pageable
// copies take 10 us each). False when the four copies have to do it: more rows than a slot holds,
// no slot free, rows of another device than the current one, or a destination that is not host
// memory.
bool copy_few_rows(const SearchOut &o, const uint32_t *order, uint32_t *q, uint32_t *e, double *tin,
                   double *tout, cudaStream_t s, ts_status *st)
{
    const uint64_t n = o.count;
    if (n == 0 || !o.q || n * ROW_BYTES > sizeof(HostSlot::stage) || !rows_here(o)) return false;
    cudaPointerAttributes pa;
    for (const void *p : {(const void *)q, (const void *)e, (const void *)tin, (const void *)tout})
        if (p && (cudaPointerGetAttributes(&pa, p) != cudaSuccess ||
                  pa.type == cudaMemoryTypeDevice)) {
            cudaGetLastError();
            return false;
        }
    struct Slot {
        HostSlot *h = g_slots.take();
        ~Slot() { if (h) g_slots.give(h); }
    } slot;
    void *d = nullptr;
    if (!slot.h || cudaHostGetDevicePointer(&d, slot.h->stage, 0) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    *st = [&]() -> ts_status {
        TS_LAUNCH_PDL(k_rows_out, dim3(nblk(n)), dim3(TPB), 0, s, n, order, o.q, o.e, o.tin,
                      o.tout, static_cast<double *>(d));
        TS_CUDA(cudaStreamSynchronize(s));
        const double *h = slot.h->stage;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(h + 2 * n);
        if (tin) memcpy(tin, h, 8 * n);
        if (tout) memcpy(tout, h + n, 8 * n);
        if (q) memcpy(q, w, 4 * n);
        if (e) memcpy(e, w + n, 4 * n);
        return TS_OK;
    }();
    return true;
}

// copy_sorted_rows on the device; *done stays false where its memory does not reach for that.
static ts_status sort_rows_here(const SearchOut &o, uint32_t *q, uint32_t *e, double *tin,
                                double *tout, cudaStream_t s, bool *done)
{
    const uint64_t n = o.count;
    const int eb = o.n_entries ? bits_for(o.n_entries - 1) : 32;
    const int qb = o.stats.n_queries ? bits_for(o.stats.n_queries - 1) : 32;
    DevBuf keys, vals, rows;
    TS_CHECK(keys.alloc(8 * n, s));
    TS_CHECK(vals.alloc(4 * n, s));
    TS_LAUNCH_PDL(k_row_keys, dim3(nblk(n)), dim3(TPB), 0, s, n, o.q, o.e, eb,
                  keys.as<uint64_t>(), vals.as<uint32_t>());
    TS_CHECK(radix_sort_u64(keys.as<uint64_t>(), vals.as<uint32_t>(), n, eb + qb, s, nullptr,
                            false));
    keys.release();
    ts_status few = TS_OK;
    *done = copy_few_rows(o, vals.as<uint32_t>(), q, e, tin, tout, s, &few);
    if (*done) return few;
    TS_CHECK(rows.alloc(ROW_BYTES * n, s));
    double *d = rows.as<double>();
    uint32_t *w = reinterpret_cast<uint32_t *>(d + 2 * n);
    TS_LAUNCH_PDL(k_rows_out, dim3(nblk(n)), dim3(TPB), 0, s, n, vals.as<uint32_t>(), o.q, o.e,
                  o.tin, o.tout, d);
    if (tin) TS_CUDA(cudaMemcpyAsync(tin, d, 8 * n, cudaMemcpyDeviceToHost, s));
    if (tout) TS_CUDA(cudaMemcpyAsync(tout, d + n, 8 * n, cudaMemcpyDeviceToHost, s));
    if (q) TS_CUDA(cudaMemcpyAsync(q, w, 4 * n, cudaMemcpyDeviceToHost, s));
    if (e) TS_CUDA(cudaMemcpyAsync(e, w + n, 4 * n, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    *done = true;
    return TS_OK;
}

// Rows to the host by (query, entry): sorted on the device (the two indices are one key of as many
// bits as queries and entries take; no two rows have the same) and copied from one block. Rows of
// another device, or more than the device's memory can sort (25 B a row, then 28 with the block of
// sorted rows), are sorted here. 15,000 rows, sorted by numpy from the host's copy before: 1147
// -> 433 us with their search.
ts_status copy_sorted_rows(const SearchOut &o, uint32_t *q, uint32_t *e, double *tin, double *tout,
                           cudaStream_t s)
{
    const uint64_t n = o.count;
    if (n == 0 || !o.q) {
        TS_CUDA(cudaStreamSynchronize(s));
        return TS_OK;
    }
    if (n <= 0xffffffffull && rows_here(o)) {
        bool done = false;
        const ts_status st = sort_rows_here(o, q, e, tin, tout, s, &done);
        if (done || (st != TS_OK && st != TS_ERR_OOM)) return st;
    }
    std::vector<uint32_t> hq(n), he(n);
    std::vector<double> ha(n), hb(n);
    TS_CUDA(cudaMemcpyAsync(hq.data(), o.q, 4 * n, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(he.data(), o.e, 4 * n, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(ha.data(), o.tin, 8 * n, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(hb.data(), o.tout, 8 * n, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    std::vector<uint64_t> at(n);
    for (uint64_t i = 0; i < n; i++) at[i] = i;
    std::sort(at.begin(), at.end(), [&](uint64_t a, uint64_t b) {
        return hq[a] != hq[b] ? hq[a] < hq[b] : he[a] < he[b];
    });
    for (uint64_t i = 0; i < n; i++) {
        if (q) q[i] = hq[at[i]];
        if (e) e[i] = he[at[i]];
        if (tin) tin[i] = ha[at[i]];
        if (tout) tout[i] = hb[at[i]];
    }
    return TS_OK;
}

// The query columns of stationary points: x0 = x1 = x (likewise y, z), t0 = t_start, t1 = t_end.
__global__ void k_point_cols(const double *x, const double *y, const double *z, uint64_t n,
                             double ts, double te, double *cols)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const double px = x[i], py = y[i], pz = z[i];
        cols[i] = px;
        cols[n + i] = py;
        cols[2 * n + i] = pz;
        cols[3 * n + i] = ts;
        cols[4 * n + i] = px;
        cols[5 * n + i] = py;
        cols[6 * n + i] = pz;
        cols[7 * n + i] = te;
    }
}

ts_status search_points(const Index *ix, const double *x, const double *y, const double *z,
                        uint64_t n, bool on_host, const ts_query_params *qp, cudaStream_t s,
                        SearchOut *out)
{
    TS_CHECK(check_query_params(qp));
    if (!(qp->t_start < qp->t_end)) {
        set_error("ts_search_points: the interval must have positive length");
        return TS_ERR_INVALID_ARG;
    }
    if (n && (!x || !y || !z)) {
        set_error("ts_search_points: NULL coordinate array");
        return TS_ERR_INVALID_ARG;
    }
    *out = SearchOut{};
    if (n == 0) return TS_OK;
    DevBuf pts, cols;
    const double *px = x, *py = y, *pz = z;
    if (on_host) {
        TS_CHECK(pts.alloc(sizeof(double) * 3 * n, s));
        double *d = pts.as<double>();
        TS_CUDA(cudaMemcpyAsync(d, x, sizeof(double) * n, cudaMemcpyHostToDevice, s));
        TS_CUDA(cudaMemcpyAsync(d + n, y, sizeof(double) * n, cudaMemcpyHostToDevice, s));
        TS_CUDA(cudaMemcpyAsync(d + 2 * n, z, sizeof(double) * n, cudaMemcpyHostToDevice, s));
        px = d;
        py = d + n;
        pz = d + 2 * n;
    }
    TS_CHECK(cols.alloc(sizeof(double) * 8 * n, s));
    k_point_cols<<<nblk(n), TPB, 0, s>>>(px, py, pz, n, qp->t_start, qp->t_end,
                                         cols.as<double>());
    TS_LAUNCHED();
    ts_segments q;
    memset(&q, 0, sizeof(q));
    const double *c = cols.as<double>();
    q.x0 = c; q.y0 = c + n; q.z0 = c + 2 * n; q.t0 = c + 3 * n;
    q.x1 = c + 4 * n; q.y1 = c + 5 * n; q.z1 = c + 6 * n; q.t1 = c + 7 * n;
    q.n = n;
    q.on_host = 0;
    // (every point's window is the interval's part of the database's time)
    const double window = std::min(qp->t_end, ix->tmax) - std::max(qp->t_start, ix->tmin);
    return search_plain(ix, &q, qp, s, out, std::max(0.0, window));
}

ts_status schedule_only(const Index *ix, const ts_segments *q, const ts_query_params *qp,
                        cudaStream_t s, int32_t *sel, uint64_t *lo, uint64_t *hi)
{
    TS_CHECK(check_query_params(qp));
    if (!q || !sel || !lo || !hi) {
        set_error("ts_schedule: NULL argument");
        return TS_ERR_INVALID_ARG;
    }
    const uint64_t nq = q->n;
    if (nq == 0) return TS_OK;
    DevBuf qcopy;
    const double *cols[8];
    TS_CHECK(device_cols(q, s, qcopy, cols));
    PlainWork w;
    PipeBufs b;
    PipeCaps c;
    TS_CHECK(plain_prepare(ix, cols, nq, qp, s, w, b, c, false));
    uint32_t st = 0;
    if (ix->kind == TS_INDEX_SPATIAL) {
        // per query: number of z-runs and of candidates (sum of the runs' lengths)
        std::vector<uint32_t> off(nq + 1), ul(c.units), uh(c.units);
        TS_CUDA(cudaMemcpyAsync(off.data(), b.quoff, 4 * (nq + 1), cudaMemcpyDeviceToHost, s));
        if (c.units) {
            TS_CUDA(cudaMemcpyAsync(ul.data(), b.u_lo, 4 * c.units, cudaMemcpyDeviceToHost, s));
            TS_CUDA(cudaMemcpyAsync(uh.data(), b.u_hi, 4 * c.units, cudaMemcpyDeviceToHost, s));
        }
        TS_CUDA(cudaMemcpyAsync(&st, b.status, 4, cudaMemcpyDeviceToHost, s));
        TS_CUDA(cudaStreamSynchronize(s));
        TS_CHECK(read_dev_status(st));
        for (uint64_t i = 0; i < nq; i++) {
            sel[i] = SEL_GRID;
            lo[i] = off[i + 1] - off[i];
            uint64_t cand = 0;
            for (uint32_t u = off[i]; u < off[i + 1]; u++) cand += uh[u] - ul[u];
            hi[i] = cand;
        }
        return TS_OK;
    }
    std::vector<uint32_t> hs(nq), hl(nq), hh(nq);
    TS_CUDA(cudaMemcpyAsync(hs.data(), b.u_sel, 4 * nq, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(hl.data(), b.u_lo, 4 * nq, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(hh.data(), b.u_hi, 4 * nq, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaMemcpyAsync(&st, b.status, 4, cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    TS_CHECK(read_dev_status(st));
    for (uint64_t i = 0; i < nq; i++) {
        sel[i] = (int32_t)hs[i];
        lo[i] = hl[i];
        hi[i] = hh[i];
    }
    return TS_OK;
}

}  // namespace ts
