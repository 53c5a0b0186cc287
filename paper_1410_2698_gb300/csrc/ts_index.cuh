// ts_index.cuh -- the resident index (Sec. 4.1-4.3 re-laid out for HBM).
#pragma once

#include <vector>

#include "ts_internal.cuh"

namespace ts {

constexpr uint32_t MAGIC_INDEX = 0x54534958u;   // "TSIX"
constexpr uint32_t MAGIC_RESULT = 0x54535253u;  // "TSRS"

struct Index {
    uint32_t magic = MAGIC_INDEX;
    int kind = 0;
    uint64_t n = 0;
    int device = 0;

    // entries in start-time order (Sec. 4.2: D sorted by t_start and renumbered)
    SegD *seg = nullptr;     // exact FP64 data
    uint32_t *orig = nullptr;  // sorted position -> caller's index

    // extents (exact, from the ingest reductions)
    double tmin = 0, tmax = 0, max_dur = 0;
    double emin[3] = {0, 0, 0}, emax[3] = {0, 0, 0}, longest[3] = {0, 0, 0};

    // the entries of every temporal bin in the order in which they are swept, near ones together
    // (MortonMap; the bins keep their ranges [B^first, B^last]): prefilter records with their
    // start-time positions, and the bounding record of every aligned chunk of 64 (built for every
    // kind whose ranges cover bins)
    Chunk *trec = nullptr;
    RecF *tbox = nullptr;
    float *axis_rank = nullptr;  // share of the entries before each of 256 places of each axis

    // temporal bins (Sec. 4.2)
    uint32_t m = 0;
    double b = 0;
    double *bin_start = nullptr, *bin_end = nullptr, *bin_pmax = nullptr;  // m each
    uint32_t *bin_off = nullptr;  // m + 1

    // spatiotemporal subbins (Sec. 4.3): per dimension an id array in (subbin, bin, sweep) order
    // (the export gives it in start-time order), a duplicated prefilter record per id, the
    // chunks' bounding records, and offsets off[j*m + i]
    uint32_t v[3] = {0, 0, 0};
    double sub_lo[3] = {0, 0, 0}, sub_w[3] = {0, 0, 0};
    uint32_t *st_ids[3] = {nullptr, nullptr, nullptr};
    Chunk *st_rec[3] = {nullptr, nullptr, nullptr};
    RecF *st_box[3] = {nullptr, nullptr, nullptr};
    uint32_t *st_off[3] = {nullptr, nullptr, nullptr};
    double *sub_bound[3] = {nullptr, nullptr, nullptr};  // lo + j*w for j = 0..v
    uint64_t st_len[3] = {0, 0, 0};

    // flatly structured grid (Sec. 4.1), one cell per entry (the cell of its MBB's minimum
    // corner): dense cell offsets over g^3 cells and the lookup array A with a copy of each
    // entry's prefilter record; inside a cell the entries keep their start-time order, so the
    // bounding records of its chunks are narrow in time
    uint32_t g = 0;
    double g_lo[3] = {0, 0, 0}, g_w[3] = {0, 0, 0};
    uint32_t *ga = nullptr;
    Chunk *ga_rec = nullptr;
    RecF *gbox = nullptr;  // bounding record of every aligned chunk of 64 of ga_rec
    uint32_t *g_off = nullptr;  // g^3 + 1
    double *g_bound[3] = {nullptr, nullptr, nullptr};  // lo + j*w for j = 0..g
    uint64_t g_len = 0;

    size_t bytes = 0;
    std::vector<void *> allocs;
    cudaStream_t stream = nullptr;  // of the build

    template <class T>
    ts_status alloc(T **p, size_t count)
    {
        size_t nb = sizeof(T) * (count ? count : 1);
        cudaError_t e = index_malloc((void **)p, nb, stream, device);
        if (e != cudaSuccess) {
            *p = nullptr;
            return cuda_status(e, "index_malloc");
        }
        allocs.push_back((void *)*p);
        bytes += nb;
        return TS_OK;
    }
};

// Morton code of a point among the database's entries: its rank along each axis (the share of the
// entries before it, from a table over the extents), `bits` bits of it, interleaved. Ranks rather
// than coordinates: entries crowd, and so do the queries, and a few bits of the coordinate leave a
// crowd in one cell (merger, 100,000 query segments of the cores: 1.20M chunks swept with 3 bits of
// the coordinates, 0.93M with 4 of the ranks; pair kernel 0.84 -> 0.69 ms, with the per-member pass
// that small chunks call for).
// Points outside (queries) take the nearest cell; the code only orders, so its FP32 rounding never
// matters.
//
// Where the occupied bins hold BY_X_ENTRIES or fewer on average, entries and queries are ordered by x
// alone. A bin's runs of 64 are slabs then, 1/N of the extent thin for N runs, where along the curve
// they are cubes of N^(-1/3) of the extent an axis that mostly straddle two cells: of few, a query
// meets more cubes than slabs. Pair kernel, slabs / cubes, us: walks 500 entries a bin 111 / 138
// (four distances, 40,000 query segments), 2,500 a bin 37 / 39, 10,000 a bin 41 / 41; dense 4,000 a
// bin 36 / 36, 20,000 a bin 237 / 196; merger 10,000 a bin 53 / 51. (Occupied: trajectories sampled
// at the same times leave most bins empty.)
constexpr int AXIS_BINS = 256;
constexpr uint64_t BY_X_ENTRIES = 4096;

struct MortonMap {
    float lo[3], inv[3];
    const float *rank;  // 3 x (AXIS_BINS + 1), and 1 where the order is that of x alone, 0 elsewhere
    int bits;

    __device__ static __forceinline__ uint32_t spread(uint32_t v)  // bit k -> bit 3k, 10 bits
    {
        v = (v | (v << 16)) & 0x030000ffu;
        v = (v | (v << 8)) & 0x0300f00fu;
        v = (v | (v << 4)) & 0x030c30c3u;
        return (v | (v << 2)) & 0x09249249u;
    }
    // place among the axis's bins, [0, AXIS_BINS) (NaN: 0)
    __device__ __forceinline__ float place(float x, int d) const
    {
        return fminf(fmaxf((x - lo[d]) * inv[d], 0.0f), (float)AXIS_BINS - 0.01f);
    }
    __device__ __forceinline__ uint32_t cell(float x, int d, int bits) const
    {
        const float p = place(x, d);
        const int k = (int)p;
        const float a = rank[d * (AXIS_BINS + 1) + k], b = rank[d * (AXIS_BINS + 1) + k + 1];
        const float r = a + (p - (float)k) * (b - a);
        return min((uint32_t)(r * (float)(1 << bits)), (1u << bits) - 1u);
    }
    __device__ __forceinline__ uint32_t code(float x, float y, float z) const
    {
        // (12 bits tell the entries of a small bin apart; a digit that is 0 in all keys sorts faster,
        // 24 us a pass over 1M keys where a random one takes 38)
        if (rank[3 * (AXIS_BINS + 1)] != 0.0f)
            return cell(x, 0, min(3 * bits, 12)) << max(3 * bits - 12, 0);
        return spread(cell(x, 0, bits)) | (spread(cell(y, 1, bits)) << 1) |
               (spread(cell(z, 2, bits)) << 2);
    }
};

inline MortonMap morton_map(const Index *ix, int bits)
{
    MortonMap m;
    m.bits = bits;
    m.rank = ix->axis_rank;
    for (int d = 0; d < 3; d++) {
        const double ext = ix->emax[d] - ix->emin[d];
        m.lo[d] = (float)ix->emin[d];
        const float inv = ext > 0.0 ? (float)((double)AXIS_BINS / ext) : 0.0f;
        m.inv[d] = inv < 3.0e38f ? inv : 0.0f;
    }
    return m;
}

}  // namespace ts
