// Internal declarations shared by the translation units of libqamw (not part of the C ABI).
#ifndef QAMW_INTERNAL_H_
#define QAMW_INTERNAL_H_

#include <cstdint>
#include <vector>

#include "qamw.h"

namespace qamw {

inline bool is_pow2(int64_t v) { return v > 0 && (v & (v - 1)) == 0; }
inline int ilog2(int64_t v) {
    int l = 0;
    while ((int64_t(1) << l) < v) ++l;
    return l;
}

// Column (and, with the same map, row) of the search grid that holds coordinate z:
//     c = min(max(z, -zmax), zmax);  t = c * c;
//     column = half + rn(c * (c0 + t * (c1 + t * c2)))            (rn: to nearest integer)
// an odd polynomial with slope a ((1 - t / T)^2 + eps): cells are narrow where a Gaussian source
// puts its codewords, widen up to sqrt(T) and get a few more columns between there and
// zmax = rho sqrt(T) for heavy-tailed inputs; the outermost columns take everything beyond.  The
// device evaluates it in f32 (three fused multiply-adds, the last one onto 1.5 * 2^23 + half, which
// leaves the integer in the low mantissa bits).  grid = 2 * half + 1 is odd.
struct CellMap {
    int grid = 0, half = 0;
    float zmax = 0.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
};
struct MapShape {
    double T = 18.0, eps = 0.02, rho = 1.25;
};
CellMap make_cell_map(int grid, const MapShape& shape);
// The map in exact arithmetic on the f32 coefficients (before rounding to an integer).
double cell_map_value(const CellMap& m, double z);

// Host form of the search grid: per cell the full candidate list.
struct CellLists {
    CellMap map;
    // Column j can be returned by the device for z in [lo[j], hi[j]]: the interval of the exact map
    // widened by a margin that covers the device's rounding; the outermost reach +-16384.
    std::vector<double> lo, hi;
    std::vector<std::vector<uint16_t>> lists;  // [iy*grid + ix], ascending codeword indices
    int max_list = 0;
    int n_candidates = 0;
};

// Device form (see pack_search_table in qamw_table.cpp).
struct SearchTable {
    CellMap map;
    std::vector<uint16_t> cells;      // grid*grid records of 4 x u16
    std::vector<uint16_t> overflow;   // candidate lists of cells with more than 4 entries
    int n_overflow_cells = 0;
    int max_list = 0;
    int n_candidates = 0;
    size_t bytes() const { return cells.size() * 2 + overflow.size() * 2; }
};

// Nearest-neighbour (Voronoi) polygons of all codewords, clipped to |z| <= 16384: the vertices of
// codeword i are xy[2 * start[i]] .. xy[2 * start[i + 1]).
struct VoronoiSet {
    std::vector<int> start;
    std::vector<double> xy;
};
void voronoi_polygons(const double* cb, int K, VoronoiSet* out);

int default_grid(int K);
bool build_cell_lists(const VoronoiSet& vs, int K, const CellMap& map, CellLists* out);
bool build_cell_lists(const double* cb, int K, int grid, CellLists* out);  // default map shape
double overflow_cost(const CellLists& cl);
bool pack_search_table(const CellLists& cl, SearchTable* out);

// grid > 0 (odd): exactly that grid (fails if it does not fit); grid == 0: `first` columns (0: the default for
// K), shrunk until the table fits in budget_bytes.
bool choose_search_table(const float* codebook, int K, int grid, size_t budget_bytes, SearchTable* out, int first = 0);
// The records as the kernels read them (SearchSmem in qamw_device.cuh), for codebook entries of 2^log2_entry bytes:
// grid * grid * 2 words, and the list words.  False if the lists do not fit their fields.
bool pack_device_table(const SearchTable& t, int K, int log2_entry, std::vector<uint32_t>* words, std::vector<uint32_t>* lists);

#ifdef __CUDACC__
#define QAMW_HOST_DEVICE __host__ __device__
#else
#define QAMW_HOST_DEVICE
#endif

// SplitMix64 finaliser (Steele, Lea, Flood 2014) and the increment of its counter: signs and Gaussian samples.
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ULL;
QAMW_HOST_DEVICE inline uint64_t mix64(uint64_t x) {
    x ^= x >> 30;
    x *= 0xBF58476D1CE4E5B9ULL;
    x ^= x >> 27;
    x *= 0x94D049BB133111EBULL;
    x ^= x >> 31;
    return x;
}
// Key of the sample stream `seed`: sample i takes counters 2i and 2i + 1.
QAMW_HOST_DEVICE inline uint64_t sample_key(uint64_t seed) { return mix64(seed ^ 0xD1B54A32D192ED03ULL); }
// Sign of column j: -1 or 1.
QAMW_HOST_DEVICE inline int8_t column_sign(uint64_t seed, int j) { return (mix64(seed + kGolden * uint64_t(j + 1)) >> 63) ? int8_t(-1) : int8_t(1); }

// The samples [lo, hi) of a cell as a warp walks them, STEP at a time.  Positions are 64-bit: a call may have up to
// 2^31 - 1 samples, so a position of the next step need not fit an int.
template <int STEP>
struct CellWalkBy {
    static constexpr int kStep = STEP;
    long long base, hi;
    QAMW_HOST_DEVICE CellWalkBy(int lo, int end) : base(lo), hi(end) {}
    QAMW_HOST_DEVICE bool more() const { return base < hi; }
    QAMW_HOST_DEVICE bool full() const { return hi - base >= kStep; }
    QAMW_HOST_DEVICE int left() const { return int(hi - base); }
    QAMW_HOST_DEVICE bool has(int k) const { return base + k < hi; }  // k < 2 kStep: this step's samples and the next one's
    QAMW_HOST_DEVICE long long at(int k) const { return base + k; }
    QAMW_HOST_DEVICE void step() { base += kStep; }
};
using CellWalk = CellWalkBy<64>;

void set_cuda_error(const char* what, int code);
void set_error_text(const char* text);

// One weight matrix as the batched (multi-matrix) kernels see it: plain device pointers and sizes.
struct MatDesc {
    const void* W;
    const float* chan_scale;
    const int8_t* signs;
    const float* sigma;
    const float* act_rms;
    uint8_t* packed;
    float* row_norm;
    void* w_hat;
    double* dist4;
    long long w_row_stride;       // elements
    long long packed_row_stride;  // bytes
    long long calib_offset;       // batched calibration: byte offset of this matrix's partial sums in the workspace,
    int calib_first_block;        //   the first block whose span touches it, and the number of slots it has
    int calib_slots;              //   (blocks touching it), each [pair_stride] doubles
    int d_out, d_in;
};

// Fast multi-matrix paths (qamw_rows.cu).  `descs` is a device array of n descriptors, or NULL with
// n == 1 and the single descriptor passed by value.  They return QAMW_ERR_SHAPE without launching
// when a matrix does not meet the fast kernels' layout rules; the caller then uses the general kernels.  With `count`
// they only add the number of their launches to it.
int rows_decode(const MatDesc* descs_dev, const MatDesc* descs_host, int n, const void* spans_dev, int span_blocks,
                int block, int K, const float* codebook_dev, uint32_t flags, void* stream, int* count = nullptr);
int rows_encode(const MatDesc* descs_dev, const MatDesc* descs_host, int n, const void* spans_dev, int span_blocks,
                int block, int K, int w_bf16, const ::qamw_codebook* cb, uint32_t flags, int32_t* status, void* stream,
                void* calib_base = nullptr,  // run the calibration pass instead (cb may be NULL)
                int* count = nullptr);
// Sign mask and, if act_host is not NULL, channel scales of the columns, on the stream (qamw_prepare.cu); act_host
// may be overwritten as soon as the call returns.
int prepare_columns(const float* act_host, int d_in, float alpha, uint64_t seed, float* chan_scale, int8_t* signs, void* stream);
// The calibration pass and its finish for one matrix; QAMW_ERR_SHAPE as above.
int rows_calibrate(MatDesc d, int block, int w_bf16, uint32_t flags, void* workspace, size_t workspace_bytes, int32_t* status,
                   void* stream);
int sm_count();
// log2 of the number of bank-separated codebook copies a block keeps in shared memory (at most 16, and at most
// `budget` bytes) when it makes `gathers` warp-wide codeword reads in all.  A copy costs its stores (one wavefront per 128
// bytes), more copies save wavefronts per read: with 16 copies a read takes 2 wavefronts, with 8, 4, 2 and 1
// about 4, 5.4, 5.9 and 6.2 (16 random lanes on 16 pairs of banks, twice).
int pick_copies(int K, long long gathers, size_t budget);
int check_matrix_params(const qamw_params* p);
long long distortion_items(int d_out, int d_in);  // work items of the distortion kernel for one matrix
// Where the blocks of the batched distortion kernel leave their partial sums: records of four doubles,
// matrix by matrix; matrix m appears in the spans of blocks owner[m].first .. owner[m].last and block b's
// record for it is number owner[m].offset + b - owner[m].first.  counter[m] counts the blocks that have left theirs;
// the last one adds the records up in a fixed order and resets it.
struct DistOwner {
    int first, last;  // blocks
    int offset;       // first record of the matrix
};
struct DistReduce {
    double* partial;
    const DistOwner* owner;
    unsigned int* counter;  // one per matrix, zero between launches
};
int distortion_batch_launch(const MatDesc* descs_dev, const void* spans_dev, int blocks, int w_bf16,
                            const DistReduce& red, void* stream);  // QAMW_OK or the error code every entry point reports

}  // namespace qamw

struct qamw_codebook {
    int K = 0;
    int device = -1;
    // one device allocation: [codebook K*2 f32][cell records grid^2 * 2 words][list words] (see pack_device_table)
    void* d_blob = nullptr;
    size_t blob_bytes = 0;
    size_t off_cells = 0, off_overflow = 0;
    int log2c = 0;  // log2 of the codebook copies that the cell records assume
    qamw::CellMap map;
    int n_candidates = 0, max_list = 0, n_overflow_cells = 0;
    std::vector<float> h_codebook;  // host copy (decode only needs the device codebook)
    // polar baseline: the blob then is [codebook K*2 f32][squared amplitude thresholds 2^Ba f32]
    // [boundary unit vectors 2^Bp / 2 float2] and off_cells / off_overflow point at the two tables
    bool polar = false;
    int polar_ba = 0, polar_bp = 0;
};

#endif  // QAMW_INTERNAL_H_
