// Codebook training on the device (Section 3.6: Lloyd iterations on the unit circular Gaussian).
//
// One iteration = an exact assignment pass (nearest codeword of every sample in double, lowest index on
// ties) and a centroid pass in which every cell's samples are added in sample order, so the sums are bit
// for bit those of a sequential loop over the samples and training gives the same codebook run after run.
//
// Assignment.  Once per call the samples are put in the order of a Hilbert curve, so that 256
// consecutive ones (a tile, one block) lie in a small box.  Per iteration a block finds the codewords that
// can be nearest to some point of its box -- those whose smallest distance to the box does not exceed the
// smallest of all largest distances -- and each of its warps narrows the list again with the box of its own 32
// samples: a sample is compared with about 3 of 2048 codewords instead of all.  The filter and the comparison run in f32 with
// bounds on their rounding; where those leave a doubt the comparison is made in double arithmetic, so the result is that of the
// exhaustive scan.
//
// Centroids.  A stable counting sort by cell (per-chunk histograms, prefix sums, a scatter that ranks
// equal keys inside a warp by lane) brings every cell's samples together in sample order.  The chain
// of additions of a cell is serial by contract.
//
// Incremental updates.  After the first eight passes few samples still change cells.  From then on the cells keep their
// samples in order, the assignment looks at a neighbourhood of each tile and reports what changes, and the update puts the changes
// in their places: two kernels in place of five, the same sums in the same order.
//
// The stopping rule is evaluated on the device: a batch of iterations is enqueued at once, the kernels
// after the last wanted update return at once, and the host reads the errors once per batch.
//
// K = 2048 on 2^20 samples, 100 updates on a B200: 235 ms with the exhaustive scan, a serial scan of the histograms
// and one host round trip per update; 8.6 with five kernels for every update; 5.3 with incremental ones (ms).
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <vector>

#include "qamw_device.cuh"
#include "qamw_internal.h"
#include "qamw_launch.h"

using namespace qamw;

namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kTile = 256;           // samples per tile, threads of its block
constexpr int kSortWarps = 16;       // warps that sort a chunk
constexpr int kMinChunk = 4096;      // samples per sorting chunk; more when there would be more than this
constexpr int kManyChunks = 1024;    // many chunks,
constexpr int kMaxChunk = 65504;     // but not more than 16-bit counters hold
constexpr int kBatch = 16;           // iterations enqueued between two looks at the stopping rule
constexpr int kFullFirst = 8;        // passes in full before the first incremental one,
constexpr int kFullAgain = 4;        // and after one that ran out of room

// Unit circular Gaussian samples by Box-Muller from the counter stream of the header: sample i uses
// the uniforms of counters 2i and 2i+1.
__global__ void sample_kernel(unsigned long long key, unsigned long long n, double2* out) {
    chain_release();
    chain_wait();
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const double u1 = (double(mix64(key + kGolden * (2 * i + 1)) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        const double u2 = (double(mix64(key + kGolden * (2 * i + 2)) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        const double rad = sqrt(-2.0 * log(u1));
        double s, c;
        sincos(6.283185307179586476925286766559 * u2, &s, &c);
        out[i] = make_double2(rad * c, rad * s);
    }
}

// What the kernels of one call share: the stopping rule's state and the errors of the current batch.
struct TrainState {
    double prev;             // mean squared distance before the last update
    double trace[kBatch];    // of the last assignments: pass t at t % kBatch
    int passes;              // assignments so far
    int updates;             // centroid updates decided on
    int done;                // the rule has been met: later kernels return at once
    // Incremental passes.  A kernel only asks for what the kernels before it have written: warps of a block that saw a flag
    // change under way would part.
    int stalled;             // the assignment has run out of room: the pass is repeated in full (written by the assignment)
    int skip;                // the update has nothing to do (written by the assignment)
    int held;                // later assignments have nothing to do until then (written by the update)
    unsigned ticket;         // blocks of the prefix kernel that have finished; zero between launches
    alignas(16) unsigned moved[kBatch];  // incremental updates since the neighbourhoods were listed: bits of the longest step of a codeword
};

// ---------------------------------------------------------------------------------------------
// spatial order of the samples (once per call)
// ---------------------------------------------------------------------------------------------

// Root mean square coordinate of the first samples.  It only decides how well the tiles are packed.
__global__ void __launch_bounds__(1024) scale_kernel(const double2* samples, unsigned long long n, float* scale) {
    chain_release();
    chain_wait();
    __shared__ float part[32];
    float s = 0.f;
    const int m = int(min(n, 4096ull));
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const float x = float(samples[i].x), y = float(samples[i].y);
        s += x * x + y * y;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(kFullMask, s, d);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 32; ++w) t += part[w];
        *scale = sqrtf(t / float(2 * m));
    }
}

// Position of every sample along a Hilbert curve over 256 x 256 cells (16 bits).  The cells are equal steps
// of a normal distribution function 1.4 times as wide as the samples': with cells of equal width one tile of
// the sparse outskirts spans half the plane and, compared with half of the codewords, takes longer than all
// others together (1128 candidates for the worst of 4096 tiles of 256 samples, K = 2048); with cells of equal mass the
// central tiles get too wide (18 candidates on average); this is between the two (10 on average, at most 335).
__global__ void hilbert_kernel(const double2* samples, unsigned long long n, const float* scale, int* key) {
    chain_release();
    chain_wait();
    const float e = *scale, inv = e > 0.f ? 1.f / (1.4f * e) : 0.f;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        int x = min(255, max(0, int(256.f * normcdff(float(samples[i].x) * inv))));
        int y = min(255, max(0, int(256.f * normcdff(float(samples[i].y) * inv))));
        int d = 0;
        for (int s = 128; s > 0; s >>= 1) {
            const int rx = (x & s) != 0, ry = (y & s) != 0;
            d += s * s * ((3 * rx) ^ ry);
            if (!ry) {  // turn the quadrant so that the curve enters it at its start
                if (rx) {
                    x = 255 - x;
                    y = 255 - y;
                }
                const int t = x;
                x = y;
                y = t;
            }
        }
        key[i] = d;
    }
}

// Centre and half extents of a box, the half extents widened by the f32 rounding of everything that is
// subtracted from the centre; a box that is not finite (or huge) is flagged by rx < 0: all codewords then
// are candidates.  For each 32 and each 64 samples, and one for the whole tile.
struct TileBox {
    float mx, my, rx, ry;
};
constexpr int kTileWarps = kTile / 32;
constexpr int kBoxes = kTileWarps + 1 + kTileWarps / 2;  // per tile: of every 32 samples, of all, of every 64
__device__ __forceinline__ TileBox make_box(double x0, double x1, double y0, double y1, bool bad) {
    TileBox b;
    b.mx = float(0.5 * (x0 + x1));
    b.my = float(0.5 * (y0 + y1));
    const double slack = 1e-6;  // 2^-20: sixteen times the rounding of one f32 operation
    b.rx = float((fmax(x1 - double(b.mx), double(b.mx) - x0) + slack * fabs(double(b.mx))) * (1.0 + slack));
    b.ry = float((fmax(y1 - double(b.my), double(b.my) - y0) + slack * fabs(double(b.my))) * (1.0 + slack));
    if (bad) b.rx = -1.f;
    return b;
}
__global__ void __launch_bounds__(kTile) box_kernel(const double2* sorted, unsigned long long n, TileBox* boxes) {
    chain_release();
    chain_wait();
    __shared__ double lo[2][kTileWarps], hi[2][kTileWarps];
    __shared__ bool bad_warp[kTileWarps];
    const unsigned long long i = blockIdx.x * (unsigned long long)kTile + threadIdx.x;
    const double2 z = sorted[min(i, n - 1)];
    const bool bad = __any_sync(kFullMask, !(fabs(z.x) < 1e15) || !(fabs(z.y) < 1e15));
    double x0 = z.x, x1 = z.x, y0 = z.y, y1 = z.y;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        x0 = fmin(x0, __shfl_xor_sync(kFullMask, x0, d));
        x1 = fmax(x1, __shfl_xor_sync(kFullMask, x1, d));
        y0 = fmin(y0, __shfl_xor_sync(kFullMask, y0, d));
        y1 = fmax(y1, __shfl_xor_sync(kFullMask, y1, d));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        lo[0][w] = x0;
        hi[0][w] = x1;
        lo[1][w] = y0;
        hi[1][w] = y1;
        bad_warp[w] = bad;
        boxes[size_t(blockIdx.x) * kBoxes + w] = make_box(x0, x1, y0, y1, bad);
    }
    __syncthreads();
    auto joint = [&](int first, int count) {
        bool b = bad_warp[first];
        double l0 = lo[0][first], h0 = hi[0][first], l1 = lo[1][first], h1 = hi[1][first];
        for (int k = first + 1; k < first + count; ++k) {
            l0 = fmin(l0, lo[0][k]);
            h0 = fmax(h0, hi[0][k]);
            l1 = fmin(l1, lo[1][k]);
            h1 = fmax(h1, hi[1][k]);
            b = b || bad_warp[k];
        }
        return make_box(l0, h0, l1, h1, b);
    };
    if (threadIdx.x == 0) boxes[size_t(blockIdx.x) * kBoxes + kTileWarps] = joint(0, kTileWarps);
    if (threadIdx.x < kTileWarps / 2) boxes[size_t(blockIdx.x) * kBoxes + kTileWarps + 1 + threadIdx.x] = joint(2 * int(threadIdx.x), 2);
}

// Bounds of the squared distance from a codeword to the points of a box, each on its safe side.
__device__ __forceinline__ void box_bounds(const TileBox& b, float2 q, float& near2, float& far2) {
    const float dx = fabsf(q.x - b.mx), dy = fabsf(q.y - b.my);
    const float nx = fmaxf(dx * (1.f - 1e-6f) - b.rx, 0.f), ny = fmaxf(dy * (1.f - 1e-6f) - b.ry, 0.f);
    const float fx = dx * (1.f + 1e-6f) + b.rx, fy = dy * (1.f + 1e-6f) + b.ry;
    near2 = (nx * nx + ny * ny) * (1.f - 1e-6f);
    far2 = (fx * fx + fy * fy) * (1.f + 1e-6f);
}
constexpr float kTiny = 1e-36f;  // squares down there are no longer relatively exact

// ---------------------------------------------------------------------------------------------
// assignment
// ---------------------------------------------------------------------------------------------

// Exact nearest codeword of a warp's 32 samples among `total` listed ones, idx(0) .. idx(total - 1), of which the nearest is known to
// be one: d = dx*dx + dy*dy in double with one rounding per operation (no fused multiply-add: the result must not depend
// on how a compiler contracts the expression), the lowest index among equal distances.
//
// The box of the warp's samples narrows the list to about three codewords in the middle of the plane and up to some
// hundreds in the outskirts.  These are compared in f32; the double comparison is left to the warps in which the
// nearest two of a sample are closer to each other than f32 can tell (a few in a thousand).  With the double comparison alone, a
// candidate took its dependent 150 clocks and the outskirts set the time of the pass.
struct WarpCandidates {
    float4 c[68];  // codeword and index, padded to a whole number of steps of four
};
// Appends the codewords of the lanes in `keep` (a ballot) from position `at` on; returns the position after them.
__device__ __forceinline__ int append(WarpCandidates& buf, int at, unsigned keep, int lane, int i, float2 w) {
    if (keep >> lane & 1u) buf.c[at + __popc(keep & ((1u << lane) - 1u))] = make_float4(w.x, w.y, __int_as_float(i), 0.f);
    return at + __popc(keep);
}
// The nearest two of the first m candidates by f32 distances, added to best, second and arg, for S samples per lane.
template <int S>
__device__ __forceinline__ void compare(WarpCandidates& buf, int m, int lane, const float (&zx)[S], const float (&zy)[S], float (&best)[S],
                                        float (&second)[S], int (&arg)[S]) {
    if (lane < 4) buf.c[m + lane] = make_float4(INFINITY, INFINITY, 0.f, 0.f);
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < m; j += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 c = buf.c[j + u];
#pragma unroll
            for (int v = 0; v < S; ++v) {
                const float dx = zx[v] - c.x, dy = zy[v] - c.y;
                const float d = dx * dx + dy * dy;
                second[v] = fminf(second[v], fmaxf(best[v], d));
                arg[v] = d < best[v] ? __float_as_int(c.z) : arg[v];
                best[v] = fminf(best[v], d);
            }
        }
    }
}
__device__ __forceinline__ double exact_dist2(double2 z, double2 w) {
    const double dx = __dsub_rn(z.x, w.x), dy = __dsub_rn(z.y, w.y);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}
// Bound of the f32 rounding in a squared distance d from a sample whose larger coordinate is m: with u = 2^-24 a
// difference is off by less than 2 u m + 3 u sqrt(d), the sum of the squares by less than u (8 m sqrt(d) + 12 d) + (4 u m)^2.
__device__ __forceinline__ float dist_slack(float d, float m) {
    float root;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(d));
    return 1e-6f * (m * root + d) + 1e-12f * m * m + kTiny;
}
// f32 tells the nearer of two squared distances best <= second.
__device__ __forceinline__ bool dist_clear(float best, float second, float m) { return second < INFINITY && second - best > 2.f * dist_slack(second, m); }

template <class Index>
__device__ __forceinline__ int warp_nearest(WarpCandidates& buf, Index idx, int total, const TileBox& b, double2 z, const double2* codebook,
                                            const float2* codebook32, double& dist) {
    const int lane = threadIdx.x & 31;
    constexpr int C = 2;  // steps of 32 whose bounds stay in registers
    int mine[C];
    float2 q[C];
    float near2[C], far2 = INFINITY;
    auto bounds = [&](int k, int& i, float2& w, float& near) {
        float far;
        i = idx(min(k, total - 1));
        w = codebook32[i];
        box_bounds(b, w, near, far);
        return far;
    };
#pragma unroll
    for (int u = 0; u < C; ++u) far2 = fminf(far2, bounds(32 * u + lane, mine[u], q[u], near2[u]));
    for (int k = 32 * C + lane; k < total; k += 32) {
        int i;
        float2 w;
        float near;
        far2 = fminf(far2, bounds(k, i, w, near));
    }
    far2 = __uint_as_float(__reduce_min_sync(kFullMask, __float_as_uint(far2)));
    const float limit = b.rx < 0.f ? INFINITY : far2 + kTiny;
    auto step = [&](int k0, int& i, float2& w) {  // the codewords of one step that can be nearest
        float near;
        if (k0 == 0) {
            i = mine[0];
            w = q[0];
            near = near2[0];
        } else if (k0 == 32) {
            i = mine[1];
            w = q[1];
            near = near2[1];
        } else {
            bounds(k0 + lane, i, w, near);
        }
        return __ballot_sync(kFullMask, k0 + lane < total && !(near > limit));
    };
    const float zx[1] = {float(z.x)}, zy[1] = {float(z.y)};
    float best[1] = {INFINITY}, second[1] = {INFINITY};
    int nearest[1] = {0}, kept = 0;
    for (int k0 = 0; k0 < total; k0 += 32) {
        int i;
        float2 w;
        const unsigned keep = step(k0, i, w);
        if (keep == 0u) continue;
        __syncwarp();  // the previous step's candidates have been read
        const int m = append(buf, 0, keep, lane, i, w);
        kept += m;
        compare(buf, m, lane, zx, zy, best, second, nearest);
    }
    const bool clear = kept == 1 || dist_clear(best[0], second[0], fmaxf(fabsf(zx[0]), fabsf(zy[0])));
    int arg = nearest[0];
    if (__all_sync(kFullMask, clear)) {
        if (kept == 1) arg = __float_as_int(buf.c[0].z);  // also for samples that compare with nothing
        dist = exact_dist2(z, codebook[arg]);
        if (!(dist < INFINITY)) {  // as the exhaustive scan, which starts from codeword 0 and an infinite distance
            dist = INFINITY;
            arg = 0;
        }
        return arg;
    }
    dist = INFINITY;
    arg = 0;
    for (int k0 = 0; k0 < total; k0 += 32) {
        int i;
        float2 w;
        unsigned keep = step(k0, i, w);
        while (keep) {
            const int from = __ffs(int(keep)) - 1;
            keep &= keep - 1;
            const int c = __shfl_sync(kFullMask, i, from);
            const double d = exact_dist2(z, codebook[c]);
            // the list is in no particular order: among equals the lowest index
            arg = d < dist ? c : d == dist ? min(arg, c) : arg;
            dist = d < dist ? d : dist;
        }
    }
    if (dist == INFINITY) arg = 0;
    return arg;
}

// The assignment with a search over the whole codebook: a tile's block lists the codewords that can be nearest to some
// point of its box, its warps narrow the list.  Also adds up the distances of the tile in a fixed
// order (a shuffle tree, then by warp).  Bound by the f32 filter over all codewords (K / 256 per thread) and
// the waits between its steps, which is why the SM is filled with small blocks (eight of 256 threads; three of
// 512: 9.06 against 8.93 ms a call at K = 2048, 12.3 against 9.8 at K = 512); both arrays come from L1/L2.
template <int PER>  // codewords per thread: K / kTile, or 1 for a smaller codebook
__global__ void __launch_bounds__(kTile, 8) assign_kernel(const double2* sorted, const int* ids, unsigned long long n,
                                                       const TileBox* boxes, const double2* codebook,
                                                       const float2* codebook32, int K, int* assign, double* tile_err,
                                                       const TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ unsigned short list[QAMW_MAX_K];
    __shared__ WarpCandidates cand[kTileWarps];
    __shared__ double warp_err[kTileWarps];
    __shared__ unsigned reach;  // bits of the smallest largest squared distance (non-negative floats order as integers)
    __shared__ int count;
    if (state && state->done) return;
    if (threadIdx.x == 0) {
        reach = 0x7f800000u;
        count = 0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long i = blockIdx.x * (unsigned long long)kTile + threadIdx.x;
    const bool live = i < n;
    const double2 z = sorted[live ? i : n - 1];
    const TileBox b = boxes[size_t(blockIdx.x) * kBoxes + kTileWarps];
    const TileBox bw = boxes[size_t(blockIdx.x) * kBoxes + warp];
    // codewords that can be nearest to a point of the tile's box
    float near2[PER], far2 = INFINITY;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        near2[u] = INFINITY;
        const int c = u * kTile + threadIdx.x;
        if (PER == 1 && c >= K) break;
        float f;
        box_bounds(b, codebook32[c], near2[u], f);
        far2 = fminf(far2, f);
    }
    const unsigned m = __reduce_min_sync(kFullMask, __float_as_uint(far2));
    if (lane == 0) atomicMin(&reach, m);
    __syncthreads();
    const float limit = b.rx < 0.f ? INFINITY : __uint_as_float(reach) + kTiny;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int c = u * kTile + threadIdx.x;
        if (!(near2[u] > limit) && (PER > 1 || c < K)) list[atomicAdd(&count, 1)] = (unsigned short)c;
    }
    __syncthreads();
    double best;
    const int arg = warp_nearest(cand[warp], [&](int k) { return int(list[k]); }, count, bw, z, codebook, codebook32, best);
    if (live && assign) assign[ids[i]] = arg;
    double err = live ? best : 0.0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) err += __shfl_xor_sync(kFullMask, err, s);
    if (lane == 0) warp_err[warp] = err;
    __syncthreads();
    if (threadIdx.x == 0) {
        double e = 0.0;
        for (int w = 0; w < kTileWarps; ++w) e += warp_err[w];
        tile_err[blockIdx.x] = e;
    }
}

// ---------------------------------------------------------------------------------------------
// stable counting sort by an integer key below `bins`
// ---------------------------------------------------------------------------------------------

// The key of element i: bits [shift, shift + 8) of key[from[i]] for the spatial order, key[i] itself (the
// cell) for the centroids.
struct KeyOf {
    const int* key;
    const int* from;  // or NULL: i itself
    int shift, mask;
    __device__ __forceinline__ int operator()(unsigned long long i) const {
        return (key[from ? (unsigned long long)from[i] : i] >> shift) & mask;
    }
};

// One block of T threads adds up the tiles' errors, in the order of a block of kRuleThreads whatever T is, and applies
// the stopping rule.
constexpr int kRuleThreads = 512;
template <int T>
__device__ __forceinline__ void apply_rule(const double* tile_err, int n_tiles, unsigned long long n, double rel_tol, int max_iters,
                                           double* part, TrainState* state) {
    constexpr int V = kRuleThreads / T;  // sums per thread
    double e[V];
#pragma unroll
    for (int v = 0; v < V; ++v) e[v] = 0.0;
    for (int i = 0; i < n_tiles; i += kRuleThreads) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int k = i + v * T + int(threadIdx.x);
            if (k < n_tiles) e[v] += tile_err[k];
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) e[v] += __shfl_xor_sync(kFullMask, e[v], s);
        if ((threadIdx.x & 31) == 0) part[(v * T + threadIdx.x) >> 5] = e[v];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double total = 0.0;
        for (int w = 0; w < kRuleThreads / 32; ++w) total += part[w];
        const double D = total / double(n);
        state->trace[state->passes++ % kBatch] = D;
        if ((state->passes > 1 && state->prev - D <= rel_tol * state->prev) || state->updates >= max_iters)
            state->done = 1;
        else
            ++state->updates;
        state->prev = D;
    }
}

// Histogram of one chunk: hist[chunk * bins + bin].  In a training pass one more block adds up the tiles'
// errors in a fixed order and applies the stopping rule, beside the others.
__global__ void __launch_bounds__(kRuleThreads) hist_kernel(KeyOf key, unsigned long long n, int chunk, int bins, int* hist,
                                                   const double* tile_err, int n_tiles, double rel_tol, int max_iters,
                                                   TrainState* state) {
    chain_release();
    chain_wait();
    extern __shared__ int h[];
    __shared__ double err_part[kRuleThreads / 32];
    if (tile_err && state->done) return;
    const unsigned long long lo = blockIdx.x * (unsigned long long)chunk, hi = min(n, lo + chunk);
    if (lo >= n) {
        apply_rule<kRuleThreads>(tile_err, n_tiles, n, rel_tol, max_iters, err_part, state);
        return;
    }
    for (int c = threadIdx.x; c < bins; c += blockDim.x) h[c] = 0;
    __syncthreads();
#pragma unroll 8
    for (unsigned long long i = lo + threadIdx.x; i < hi; i += blockDim.x) atomicAdd(&h[key(i)], 1);
    __syncthreads();
    for (int c = threadIdx.x; c < bins; c += blockDim.x) hist[size_t(blockIdx.x) * bins + c] = h[c];
}

// Exclusive sum of v over the block's 1024 threads in thread order; `total` gets the sum of all.
__device__ __forceinline__ int block_scan(int v, int* warp_part, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFullMask, x, d);
        if (lane >= d) x += y;
    }
    __syncthreads();  // warp_part of the previous call has been read
    if (lane == 31) warp_part[warp] = x;
    __syncthreads();
    int p = warp_part[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFullMask, p, d);
        if (lane >= d) p += y;
    }
    total = __shfl_sync(kFullMask, p, 31);
    const int before = __shfl_sync(kFullMask, p, (warp + 31) & 31);
    return x - v + (warp ? before : 0);
}

// Prefix sums of the histograms over the chunks, bin by bin, in place: 32 bins (lanes: coalesced rows of the
// histogram) by 32 runs of chunks (warps) per block.  The block that finishes last turns the bins'
// totals into start positions.
__global__ void __launch_bounds__(1024) prefix_kernel(int* hist, int n_chunks, int bins, int* start, TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ int run_sum[32][33];
    __shared__ int warp_part[32];
    __shared__ bool last;
    if (state->done) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int bin = blockIdx.x * 32 + lane;
    const int per = (n_chunks + 31) / 32, k0 = warp * per, k1 = min(n_chunks, k0 + per);
    int sum = 0;
    if (bin < bins) {
#pragma unroll 8
        for (int k = k0; k < k1; ++k) sum += hist[size_t(k) * bins + bin];
    }
    run_sum[warp][lane] = sum;
    __syncthreads();
    if (bin < bins) {
        int before = 0;
        for (int w = 0; w < warp; ++w) before += run_sum[w][lane];
        if (warp == 31) start[bin] = before + sum;  // the bin's total, for the last block
#pragma unroll 8
        for (int k = k0; k < k1; ++k) {
            const int v = hist[size_t(k) * bins + bin];
            hist[size_t(k) * bins + bin] = before;
            before += v;
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&state->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    int carry = 0;
    for (int base = 0; base < bins; base += 1024) {
        const int c = base + int(threadIdx.x);
        const int v = c < bins ? __ldcg(start + c) : 0;
        int total;
        const int before = block_scan(v, warp_part, total);
        if (c < bins) start[c] = carry + before;
        carry += total;
    }
    if (threadIdx.x == 0) {
        start[bins] = carry;
        state->ticket = 0;
    }
}

// Stable scatter of one chunk by 16 warps, each on a contiguous run of it.  A warp walks its run 32
// elements at a time: lanes with the same key are ranked by lane, after the elements of that key which the warp
// has met before (its own counters).  The counters are then summed over the warps, key by key, and every
// element goes to: start of its key + the chunks before + the warps before + its rank.  (One warp per chunk
// of 2048 took 36 us for 2^20 samples, bound by its chain of 64 match-and-count steps; this takes 21 us, bound by
// the latency of its few steps and by scattered 16-byte stores.)
// ids_out[pos] = the element's sample number, z_out[pos] = its sample (either may be NULL).
__global__ void __launch_bounds__(32 * kSortWarps) scatter_kernel(KeyOf key, unsigned long long n, int chunk, int bins,
                                                                  const int* hist, const int* start, const double2* samples,
                                                                  int* ids_out, double2* z_out, const TrainState* state) {
    chain_release();
    chain_wait();
    extern __shared__ int cursor[];  // [bins], then 16-bit counters [warp][bins + 1 rounded up to an even number]
    if (state && state->done) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = (bins + 1) & ~1;  // counters of a warp: whole 32-bit words
    unsigned* words = reinterpret_cast<unsigned*>(cursor + bins);
    unsigned short* count = reinterpret_cast<unsigned short*>(words) + size_t(warp) * row;
    const unsigned long long c0 = blockIdx.x * (unsigned long long)chunk, c1 = min(n, c0 + chunk);
    const int run = ((chunk + kSortWarps - 1) / kSortWarps + 31) & ~31;
    const unsigned long long lo = min(c1, c0 + (unsigned long long)warp * run), hi = min(c1, lo + run);
    constexpr int U = 8;  // elements per lane that stay in registers between the two walks
    const bool keep = run <= 32 * U;
    int k[U], rank[U];
    auto load = [&](unsigned long long base) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned long long i = base + 32 * u + lane;
            k[u] = i < hi ? key(i) : -1 - lane;  // dead lanes get keys of their own
        }
    };
    auto rank_all = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned peers = __match_any_sync(kFullMask, k[u]);
            const int below = __popc(peers & ((1u << lane) - 1u));
            int seen = 0;
            if (k[u] >= 0) seen = count[k[u]];
            __syncwarp();
            if (k[u] >= 0 && below == 0) count[k[u]] = (unsigned short)(seen + __popc(peers));
            __syncwarp();
            rank[u] = seen + below;
        }
    };
    if (keep) load(lo);  // these loads travel while the counters are set up
    for (int c = threadIdx.x; c < bins; c += blockDim.x) cursor[c] = start[c] + hist[size_t(blockIdx.x) * bins + c];
    for (int c = threadIdx.x; c < kSortWarps * row / 2; c += blockDim.x) words[c] = 0u;
    __syncthreads();
    for (unsigned long long base = lo; base < hi; base += 32 * U) {
        if (!keep) load(base);
        rank_all();
    }
    __syncthreads();
    for (int w2 = threadIdx.x; w2 < row / 2; w2 += blockDim.x) {  // exclusive sums over the warps, two keys at a time
        unsigned before = 0u;  // no carry between the halves: a chunk has fewer than 65536 elements
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const unsigned v = words[w * (row / 2) + w2];
            words[w * (row / 2) + w2] = before;
            before += v;
        }
    }
    __syncthreads();
    for (unsigned long long base = lo; base < hi; base += 32 * U) {
        if (!keep) {  // a long run: its keys and ranks come once more, counted on from the sums
            load(base);
            rank_all();
        }
        constexpr int V = 4;  // samples in flight per lane
#pragma unroll
        for (int u0 = 0; u0 < U; u0 += V) {
            int id[V];
            double2 z[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const unsigned long long i = base + 32 * (u0 + v) + lane;
                id[v] = k[u0 + v] >= 0 ? (key.from ? key.from[i] : int(i)) : 0;
            }
            if (z_out) {
#pragma unroll
                for (int v = 0; v < V; ++v) z[v] = samples[id[v]];
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int kk = k[u0 + v];
                if (kk < 0) continue;
                const int pos = cursor[kk] + rank[u0 + v] + (keep ? count[kk] : 0);
                if (ids_out) ids_out[pos] = id[v];
                if (z_out) z_out[pos] = z[v];
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// centroids
// ---------------------------------------------------------------------------------------------

// Sum of the samples of one cell, samples[lo] to samples[hi - 1], in this order, by a block of 1 + LOADERS
// warps: the others bring kStage samples at a time to shared memory, by turns, two lanes of the first add up x and
// y.  The additions are one serial chain per coordinate by contract.  Returns the sum of coordinate `threadIdx.x` in threads 0 and 1.
//
// A dependent addition in registers takes 8 clocks (measured), one of this loop 9 to 10 where a block has an SM for itself; with
// one warp that both fetched and added, 64 samples at a time, 11 to 12: K = 64 on 2^20 samples took 25.1 ms, 21.3 now.
constexpr int kCellThreads = 128;  // of an incremental update
constexpr int kStage = 128;        // samples per step
struct CellStage {
    double v[2][2][kStage];  // [step parity][coordinate]
};
template <int LOADERS>
__device__ __forceinline__ double cell_sum(CellStage& st, const double2* samples, int lo, int hi) {
    constexpr int U = kStage / 32;
    const int lane = threadIdx.x & 31, loader = int(threadIdx.x >> 5) - 1;  // -1: the adder
    double2 z[U];
    CellWalkBy<kStage> walk(lo, hi), mine(lo, hi);  // the step that is added, and the loader's next one
    auto fetch = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u) z[u] = mine.has(32 * u + lane) ? samples[mine.at(32 * u + lane)] : make_double2(0.0, 0.0);
    };
    auto put = [&](int parity) {  // the loader whose step is the next one hands it over and fetches its own next one
#pragma unroll
        for (int u = 0; u < U; ++u) {
            st.v[parity][0][32 * u + lane] = z[u].x;
            st.v[parity][1][32 * u + lane] = z[u].y;
        }
#pragma unroll
        for (int w = 0; w < LOADERS; ++w) mine.step();
        fetch();
    };
    if (loader >= 0) {
        for (int w = 0; w < loader; ++w) mine.step();
        fetch();
    }
    if (loader == 0) put(0);
    __syncthreads();
    double sum = 0.0;
    for (int parity = 0; walk.more(); walk.step(), parity ^= 1) {
        if (loader >= 0) {  // the other buffer was read in the step before
            if (mine.base == walk.base + kStage) put(parity ^ 1);
        } else if (lane < 2) {
            const double* x = st.v[parity][lane];
            if (walk.full()) {
                const double2* v = reinterpret_cast<const double2*>(x);
                double2 q[2][8];
#pragma unroll
                for (int k = 0; k < 8; ++k) q[0][k] = v[k];
#pragma unroll
                for (int g = 0; g < kStage / 16; ++g) {
                    if (g + 1 < kStage / 16) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) q[(g + 1) & 1][k] = v[8 * (g + 1) + k];
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        sum += q[g & 1][k].x;
                        sum += q[g & 1][k].y;
                    }
                }
            } else {
                const int left = walk.left();
#pragma unroll 8
                for (int k = 0; k < left; ++k) sum += x[k];
            }
        }
        __syncthreads();
    }
    return sum;
}

// New codewords from the samples sorted by cell; an empty cell keeps its codeword.  The pass lasts as long as the chain
// of its largest cell.  A trained codebook's largest cells, at the centre, hold twice the mean, 2 n / K.
__global__ void __launch_bounds__(64) centroid_kernel(const double2* by_cell, const int* start, double2* codebook,
                                                                float2* codebook32, const TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ __align__(16) CellStage stage;
    if (state->done) return;
    const int c = blockIdx.x;
    const int lo = start[c], hi = start[c + 1];
    if (hi <= lo) return;
    const double sum = cell_sum<1>(stage, by_cell, lo, hi);
    if (threadIdx.x < 2) {
        const double m = sum / double(hi - lo);
        reinterpret_cast<double*>(codebook)[2 * c + threadIdx.x] = m;
        reinterpret_cast<float*>(codebook32)[2 * c + threadIdx.x] = float(m);
    }
}

// ---------------------------------------------------------------------------------------------
// incremental updates
// ---------------------------------------------------------------------------------------------

// After a few updates the codebook moves little and few samples change cells (2^20 samples, K = 2048: 17 % in the second
// pass, 2 % in the tenth, 0.1 % in the hundredth).  Each cell then keeps its samples' numbers in ascending order, the
// assignment reports the samples that change cells, and two kernels make an update instead of five: no sort, no
// candidate search over the whole codebook.  Assignment and sums are those of the full pass, bit for bit.
struct Increments {
    unsigned short* cur;      // cell of every sample, in spatial order
    unsigned short* near;     // per tile: the codewords of its neighbourhood
    int* near_n;              // per tile: how many; -1: compare with the whole codebook
    float* near_gap;          // per tile: no codeword outside the list was nearer to the tile's box than this
    int* members[2];          // sample numbers of the cells, ascending, in the slots slab[c] .. slab[c + 1) of cell c,
    double2* values[2];       //   and the samples
    int* order;               // the cells by falling size: the longest chains start first
    unsigned char* which;     // per cell: which of the two holds its present list
    int* size;                // per cell: samples
    int* slab;                // per cell: first slot
    int *arrived, *left;      // per cell: samples that have come and gone in this pass, in no particular order,
    int *n_arrived, *n_left;  //   and how many; zero between passes
};
constexpr int kNear = 64;      // codewords in a neighbourhood, if its box is not wider than that;
constexpr int kNearMost = 1024;  // such a box has up to this many
// Neighbourhoods are listed anew every so many updates (5 and 11 full passes at the start, 8 or 16 updates to a list: within 2 %).
constexpr int kEarly = 24, kNearEarly = 4, kNearLate = 8;
// Cells of up to 1024 + 2 K samples on average (37.7 million at K = 4096: slots are numbered in 32 bits), from 64 cells on: larger and fewer cells leave the merge to a few blocks, and their chains take
// the time either way.  ms a call in full and incremental: K = 64 on 70001 samples 3.9, 3.2; 128 on 70001 3.7, 2.5, on 2^18 5.2, 5.7 (5.2 in full
// is kept); 256 on 2^18 4.9, 3.7, on 2^20 10.6, 12.3; 512 on 2^20 9.5, 7.6; 2048 on 2^20 8.6, 5.3; 4096 on 2^20 10.9, 6.9.
constexpr int kIncrementalK = 64;
constexpr int kChanges = 512;  // arrivals, and departures, of a cell in one pass

// Cells as the full pass left them: members and room to grow by a quarter and `room`.
__global__ void __launch_bounds__(256) adopt_kernel(const int* by_cell, const double2* values, const int* start, int room, Increments inc, const TrainState* state) {
    chain_release();
    chain_wait();
    if (state->done) return;
    const int c = blockIdx.x, lo = start[c], hi = start[c + 1];
    const int at = lo + lo / 4 + room * c;
    for (int k = threadIdx.x; k < hi - lo; k += blockDim.x) {
        inc.members[0][at + k] = by_cell[lo + k];
        inc.values[0][at + k] = values[lo + k];
    }
    if (threadIdx.x == 0) {
        inc.which[c] = 0;
        inc.size[c] = hi - lo;
        inc.slab[c] = at;
        if (c == int(gridDim.x) - 1) inc.slab[c + 1] = hi + hi / 4 + room * (c + 1);
        inc.n_arrived[c] = inc.n_left[c] = 0;
    }
    int larger = 0;
    for (int k = threadIdx.x; k < int(gridDim.x); k += blockDim.x) {
        const int n = start[k + 1] - start[k];
        larger += n > hi - lo || (n == hi - lo && k < c);
    }
    larger = __reduce_add_sync(kFullMask, larger);
    __shared__ int part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = larger;
    __syncthreads();
    if (threadIdx.x == 0) {
        int rank = 0;
        for (int w = 0; w < 8; ++w) rank += part[w];
        inc.order[rank] = c;
    }
}

// The neighbourhood of every tile: the codewords nearest to its box, as many as fit kNear, and the distance of the
// nearest one that is left out.  While the codewords have moved by less than what separates that from the tile's
// nearest one, no other can be nearest to any of its samples.
template <int PER>
__global__ void __launch_bounds__(kTile) near_kernel(const int* ids, unsigned long long n, const TileBox* boxes, const float2* codebook32, int K,
                                                     const int* assign, Increments inc, TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ unsigned reach, gap;  // bits of non-negative floats, which order as integers
    __shared__ int count[kTileWarps], listed;
    if (state->done) return;
    if (threadIdx.x == 0) {
        reach = gap = 0x7f800000u;
        listed = 0;
        if (blockIdx.x == 0)
            for (int t = 0; t < kBatch; ++t) state->moved[t] = 0u;
    }
    if (assign) {
        const unsigned long long i = blockIdx.x * (unsigned long long)kTile + threadIdx.x;
        if (i < n) inc.cur[i] = (unsigned short)assign[ids[i]];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const TileBox b = boxes[size_t(blockIdx.x) * kBoxes + kTileWarps];
    float near2[PER], far2 = INFINITY;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        near2[u] = INFINITY;
        const int c = u * kTile + threadIdx.x;
        if (PER == 1 && c >= K) break;
        float f;
        box_bounds(b, codebook32[c], near2[u], f);
        far2 = fminf(far2, f);
    }
    const unsigned m = __reduce_min_sync(kFullMask, __float_as_uint(far2));
    if (lane == 0) atomicMin(&reach, m);
    __syncthreads();
    const float limit = __uint_as_float(reach) + kTiny;
    auto within = [&](float t) {  // codewords no farther than sqrt(t)
        int k = 0;
#pragma unroll
        for (int u = 0; u < PER; ++u) k += near2[u] <= t;
        k = __reduce_add_sync(kFullMask, k);
        __syncthreads();
        if (lane == 0) count[warp] = k;
        __syncthreads();
        k = 0;
#pragma unroll
        for (int w = 0; w < kTileWarps; ++w) k += count[w];
        return k;
    };
    float t = 2.25f * limit;  // half as far again as what can be nearest now, and more where that gives few
    int k = within(t);
    for (int round = 0; round < 24 && k < kNear && k < K; ++round) {
        const int more = within(1.4f * t);
        if (more > kNear) break;
        t *= 1.4f;
        k = more;
    }
    const bool all = b.rx < 0.f || !(limit < INFINITY) || k > kNearMost;
    float g = INFINITY;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int c = u * kTile + threadIdx.x;
        if (PER == 1 && c >= K) break;
        if (near2[u] <= t) {
            if (!all) inc.near[size_t(blockIdx.x) * kNearMost + atomicAdd(&listed, 1)] = (unsigned short)c;
        } else {
            g = fminf(g, near2[u]);  // a coordinate that is not a number leaves g alone, and such a codeword is never nearest
        }
    }
    const unsigned gm = __reduce_min_sync(kFullMask, __float_as_uint(g));
    if (lane == 0) atomicMin(&gap, gm);
    __syncthreads();
    if (!all && threadIdx.x < kNear && int(threadIdx.x) >= k)  // a whole step of them can be read
        inc.near[size_t(blockIdx.x) * kNearMost + threadIdx.x] = inc.near[size_t(blockIdx.x) * kNearMost];
    if (threadIdx.x == 0) {
        inc.near_n[blockIdx.x] = all ? -1 : k;
        inc.near_gap[blockIdx.x] = sqrtf(__uint_as_float(gap)) * (1.f - 1e-6f);
    }
}

// The assignment from the neighbourhoods: bounds of the listed codewords against the box of a warp's 64
// samples, two codewords per lane, then the comparison of assign_kernel with those that remain (about 3 of 64), two samples
// per lane.  A wide tile's longer list goes through shared memory first.  A warp whose neighbourhood may no longer be complete takes the whole
// codebook.  Samples that change cells are reported to both.
//
// Bound by the latency of three dependent loads and by issue slots (470 instructions per 64 samples, 30 % of the slots).
// 2^20 samples, K = 2048: 17 us, where assign_kernel takes 28.  Tiles that leave their blocks early do not wait for the wide ones: blocks that
// stayed and walked several tiles took longer.
constexpr int kNearThreads = kTile / 2;
__global__ void __launch_bounds__(kNearThreads, 9) near_assign_kernel(const double2* sorted, const int* ids, unsigned long long n,
                                                                      const TileBox* boxes, const double2* codebook,
                                                                      const float2* codebook32, int K, Increments inc,
                                                                      double* tile_err, TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ WarpCandidates cand[kNearThreads / 32];
    __shared__ double warp_err[kTileWarps];
    __shared__ float4 wide[kNearMost];  // a long list: codewords and their numbers
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tile = blockIdx.x;
    const unsigned long long i = tile * (unsigned long long)kTile + 64 * warp + lane;
    // everything that depends on nothing
    const int over = state->done | state->held;
    double2 z[2];
    int old[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        z[v] = sorted[min(i + 32 * v, n - 1)];
        old[v] = inc.cur[min(i + 32 * v, n - 1)];
    }
    const TileBox box = boxes[size_t(tile) * kBoxes + kTileWarps + 1 + warp];
    const unsigned short* list = inc.near + size_t(tile) * kNearMost;
    const unsigned two = reinterpret_cast<const unsigned*>(list)[lane];  // two codewords of the list
    const int total = inc.near_n[tile];
    const float gap = inc.near_gap[tile];
    float moved = 0.f;
#pragma unroll
    for (int t = 0; t < kNearLate / 4; ++t) {
        const float4 v = reinterpret_cast<const float4*>(state->moved)[t];
        moved += (v.x + v.y) + (v.z + v.w);
    }
    if (over) {
        if (tile == 0 && threadIdx.x == 0) state->skip = 1;
        return;
    }
    // no codeword outside the list is nearer to the tile's box than this by now (squared); rounding: a few units of 2^-24 each
    float reach = fmaxf(gap * (1.f - 1e-5f) - moved * (1.f + 1e-5f), 0.f);
    reach = reach * reach * (1.f - 1e-5f);
    const float zx[2] = {float(z[0].x), float(z[1].x)}, zy[2] = {float(z[0].y), float(z[1].y)};
    float best32[2] = {INFINITY, INFINITY}, second[2] = {INFINITY, INFINITY};
    float far2 = INFINITY;  // of the nearest codeword to the box
    int arg[2] = {0, 0}, kept = 0;
    double best[2] = {INFINITY, INFINITY};
    // f32 has told the nearest of all samples of the warp (see warp_nearest), or there is only one; otherwise starts over
    auto settled = [&]() {
        bool clear = true;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            if (kept == 1) arg[v] = __float_as_int(cand[warp].c[0].z);
            clear = clear && (kept == 1 || dist_clear(best32[v], second[v], fmaxf(fabsf(zx[v]), fabsf(zy[v]))));
        }
        clear = __all_sync(kFullMask, clear);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            if (clear) best[v] = exact_dist2(z[v], codebook[arg[v]]);
            else arg[v] = 0;
        }
        return clear;
    };
    auto weigh = [&](int c) {
        const double2 w = codebook[c];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const double d = exact_dist2(z[v], w);
            arg[v] = d < best[v] ? c : d == best[v] ? min(arg[v], c) : arg[v];
            best[v] = d < best[v] ? d : best[v];
        }
    };
    // Among the codewords w(0) .. w(count - 1), each with its number: their bounds against the warp's box, then those that remain.
    auto search = [&](auto w, int count, bool complete) {
#pragma unroll 8
        for (int k = lane; k < count; k += 32) {
            float near, far;
            const float4 c = w(k);
            box_bounds(box, make_float2(c.x, c.y), near, far);
            far2 = fminf(far2, far);
        }
        far2 = __uint_as_float(__reduce_min_sync(kFullMask, __float_as_uint(far2)));
        if (!complete && !(far2 < reach && box.rx >= 0.f)) {
            far2 = INFINITY;
            return false;
        }
        const float limit = box.rx >= 0.f ? far2 + kTiny : INFINITY;
        for (int k0 = 0; k0 < count; k0 += 64) {
            unsigned keep[2];
            float4 c[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = k0 + 32 * u + lane;
                c[u] = w(min(k, count - 1));
                float near, far;
                box_bounds(box, make_float2(c[u].x, c[u].y), near, far);
                keep[u] = __ballot_sync(kFullMask, k < count && !(near > limit));
            }
            if ((keep[0] | keep[1]) == 0u) continue;
            __syncwarp();
            int m = 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) m = append(cand[warp], m, keep[u], lane, __float_as_int(c[u].z), make_float2(c[u].x, c[u].y));
            kept += m;
            compare(cand[warp], m, lane, zx, zy, best32, second, arg);
        }
        if (settled()) return true;
        for (int k0 = 0; k0 < count; k0 += 32) {  // what remained, in double
            const float4 c = w(min(k0 + lane, count - 1));
            float near, far;
            box_bounds(box, make_float2(c.x, c.y), near, far);
            for (unsigned keep = __ballot_sync(kFullMask, k0 + lane < count && !(near > limit)); keep; keep &= keep - 1)
                weigh(__shfl_sync(kFullMask, __float_as_int(c.z), __ffs(int(keep)) - 1));
        }
        return true;
    };
    bool found = false;
    if (total > kNear) {
        for (int k = threadIdx.x; k < total; k += kNearThreads) {
            const int c = list[k];
            const float2 w = codebook32[c];
            wide[k] = make_float4(w.x, w.y, __int_as_float(c), 0.f);
        }
        __syncthreads();
        found = search([&](int k) { return wide[k]; }, total, false);
    } else if (total > 0) {
        const int c0 = int(two & 0xffffu), c1 = int(two >> 16);
        const float2 w0 = codebook32[c0], w1 = codebook32[c1];
        float near0, near1, far0, far1;
        box_bounds(box, w0, near0, far0);
        box_bounds(box, w1, near1, far1);
        const float f = __uint_as_float(__reduce_min_sync(kFullMask, __float_as_uint(fminf(far0, far1))));
        if (f < reach && box.rx >= 0.f) {
            found = true;
            const unsigned keep0 = __ballot_sync(kFullMask, 2 * lane < total && near0 <= f + kTiny);
            const unsigned keep1 = __ballot_sync(kFullMask, 2 * lane + 1 < total && near1 <= f + kTiny);
            kept = append(cand[warp], append(cand[warp], 0, keep0, lane, c0, w0), keep1, lane, c1, w1);
            compare(cand[warp], kept, lane, zx, zy, best32, second, arg);
            if (!settled())
                for (int k = 0; k < kept; ++k) weigh(__float_as_int(cand[warp].c[k].z));
        }
    }
    if (!found)
        search([&](int k) { const float2 w = codebook32[k]; return make_float4(w.x, w.y, __int_as_float(k), 0.f); }, K, true);
#pragma unroll
    for (int v = 0; v < 2; ++v)
        if (!(best[v] < INFINITY)) {  // as the exhaustive scan, which starts from codeword 0 and an infinite distance
            best[v] = INFINITY;
            arg[v] = 0;
        }
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        const int to = arg[v], from = old[v];
        if (i + 32 * v >= n) {
            best[v] = 0.0;
        } else if (to != from) {
            inc.cur[i + 32 * v] = (unsigned short)to;
            const int id = ids[i + 32 * v];
            const int come = atomicAdd(inc.n_arrived + to, 1), gone = atomicAdd(inc.n_left + from, 1);
            if (come < kChanges) inc.arrived[size_t(to) * kChanges + come] = id;
            if (gone < kChanges) inc.left[size_t(from) * kChanges + gone] = id;
            if (come >= kChanges || gone >= kChanges || inc.size[to] + come >= inc.slab[to + 1] - inc.slab[to]) state->stalled = 1;
        }
    }
    // the sums of assign_kernel: a shuffle tree over every 32 samples (the lower half of the warp goes on with the first 32, the
    // upper half with the others), then in order
    const double send = lane < 16 ? best[1] : best[0];
    double err = (lane < 16 ? best[0] : best[1]) + __shfl_xor_sync(kFullMask, send, 16);
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) err += __shfl_xor_sync(kFullMask, err, s);
    if ((lane & 15) == 0) warp_err[2 * warp + (lane >> 4)] = err;
    __syncthreads();
    if (threadIdx.x == 0) {
        double e = 0.0;
        for (int w = 0; w < kTileWarps; ++w) e += warp_err[w];
        tile_err[tile] = e;
    }
}

// Elements of the ascending list a[0 .. n) that are less than x.
__device__ __forceinline__ int lower_bound(const int* a, int n, int x) {
    int lo = 0;
    while (n > 0) {
        const int h = n >> 1;
        const bool right = a[lo + h] < x;
        lo += right ? h + 1 : 0;
        n = right ? n - h - 1 : h;
    }
    return lo;
}

// One block per cell: drops the samples that have left from its list, puts the new ones in their places and adds the
// cell up in the order of the list; the new codeword goes to the other copy of the codebook.  The first
// block applies the stopping rule meanwhile: if it is met, the copy that this pass has read is the result.
// Bound by its longest cells: 1160 members at K = 2048 on 2^20 samples take 1 us to find what has changed, 1 to sort it, 4 to 6 to
// place the members, 6.6 for the chain of additions (11.5 clocks each); the pass takes 18 us, where histograms, prefix sums, scatter and
// centroids take 55.  The samples move with their numbers: gathered by number instead, they kept the load/store unit busy
// (one line per lane) and an addition took 21 to 24 clocks.
__global__ void __launch_bounds__(kCellThreads, 7) update_kernel(const double2* samples, unsigned long long n, Increments inc,
                                                              const double2* codebook, double2* codebook_next, float2* codebook32_next,
                                                              const double* tile_err, int n_tiles, double rel_tol, int max_iters,
                                                              int slot, TrainState* state) {
    chain_release();
    chain_wait();
    constexpr int kChunk = 1024, kOwn = kChunk / kCellThreads, kDropped = 1 << 16;
    auto spread = [](int k) { return k + k / kOwn; };  // a thread's own members lie on a bank of its own
    struct Marks {
        int member[kChunk + kCellThreads], mark[kChunk + kCellThreads];
    };
    __shared__ __align__(16) unsigned char room[sizeof(Marks) > sizeof(CellStage) ? sizeof(Marks) : sizeof(CellStage)];
    Marks& marks = *reinterpret_cast<Marks*>(room);
    CellStage& stage = *reinterpret_cast<CellStage*>(room);
    __shared__ int come[kChanges], gone[kChanges], warp_sum[kCellThreads / 32];
    static_assert(2 * kChanges * sizeof(int) <= sizeof(room), "the changes as they come");
    const bool stalled = state->stalled;
    if (state->skip || stalled) {
        if (blockIdx.x == 0 && threadIdx.x == 0 && stalled) state->held = 1;
        return;
    }
    if (blockIdx.x == 0) {
        apply_rule<kCellThreads>(tile_err, n_tiles, n, rel_tol, max_iters, reinterpret_cast<double*>(&stage), state);
        return;
    }
    const int c = inc.order[blockIdx.x - 1];
    const int na = inc.n_arrived[c], nl = inc.n_left[c], nc = inc.size[c], which = inc.which[c], slab = inc.slab[c];
    const double2 before = codebook[c];
    if (na == 0 && nl == 0) {  // the same samples in the same order
        if (threadIdx.x == 0) {
            codebook_next[c] = before;
            codebook32_next[c] = make_float2(float(before.x), float(before.y));
        }
        return;
    }
    const int count = nc - nl + na;
    const int* old = (which ? inc.members[1] : inc.members[0]) + slab;
    int* now = (which ? inc.members[0] : inc.members[1]) + slab;
    const double2* old_values = (which ? inc.values[1] : inc.values[0]) + slab;
    double2* now_values = (which ? inc.values[0] : inc.values[1]) + slab;
    int first[kOwn];  // the front of the list is on its way while the changes are sorted
#pragma unroll
    for (int u = 0; u < kOwn; ++u) first[u] = kCellThreads * u + int(threadIdx.x) < nc ? old[kCellThreads * u + threadIdx.x] : 0;
    // the changes in ascending order: every element goes to the place that the smaller ones leave it
    {
        int* raw = reinterpret_cast<int*>(room);  // [2][kChanges]
        for (int k = threadIdx.x; k < na; k += kCellThreads) raw[k] = inc.arrived[size_t(c) * kChanges + k];
        for (int k = threadIdx.x; k < nl; k += kCellThreads) raw[kChanges + k] = inc.left[size_t(c) * kChanges + k];
        __syncthreads();
        for (int k = threadIdx.x; k < na; k += kCellThreads) {
            int r = 0;
#pragma unroll 4
            for (int j = 0; j < na; ++j) r += raw[j] < raw[k];
            come[r] = raw[k];
        }
        for (int k = threadIdx.x; k < nl; k += kCellThreads) {
            int r = 0;
#pragma unroll 4
            for (int j = 0; j < nl; ++j) r += raw[kChanges + j] < raw[kChanges + k];
            gone[r] = raw[kChanges + k];
        }
    }
    // The list, kChunk members at a time: every change finds its place among them and marks it, a sum over the marks says
    // how far each member moves.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int a0 = 0, g0 = 0;  // changes that belong before this chunk
    for (int base = 0; base == 0 || base < nc; base += kChunk) {
        const int len = min(kChunk, nc - base);
        const bool end = base + len == nc;
        __syncthreads();  // the chunk before has been written out; the changes are sorted
#pragma unroll
        for (int u = 0; u < kOwn; ++u) {
            const int k = kCellThreads * u + threadIdx.x;
            if (base) first[u] = k < len ? old[base + k] : 0;
            marks.member[spread(k)] = first[u];
            marks.mark[spread(k)] = 0;
        }
        __syncthreads();
        auto place = [&](int id) {  // members of the chunk that are less than id
            int lo = 0, m = len;
            while (m > 0) {
                const int h = m >> 1;
                const bool right = marks.member[spread(lo + h)] < id;
                lo += right ? h + 1 : 0;
                m = right ? m - h - 1 : h;
            }
            return lo;
        };
        const int top = len > 0 ? marks.member[spread(len - 1)] : 0;
        const int a1 = end ? na : lower_bound(come, na, top), g1 = end ? nl : lower_bound(gone, nl, top + 1);
        for (int j = a0 + threadIdx.x; j < a1; j += kCellThreads) {
            const int at = place(come[j]), to = base + at - lower_bound(gone, nl, come[j]) + j;
            if (at < len) atomicAdd(&marks.mark[spread(at)], 1);
            now[to] = come[j];
            now_values[to] = samples[come[j]];
        }
        for (int j = g0 + threadIdx.x; j < g1; j += kCellThreads) atomicAdd(&marks.mark[spread(place(gone[j]))], kDropped);
        __syncthreads();
        int sum = 0;  // arrivals in the lower half, departures in the upper
#pragma unroll
        for (int u = 0; u < kOwn; ++u) sum += marks.mark[spread(kOwn * threadIdx.x + u)];
        int scan = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(kFullMask, scan, d);
            if (lane >= d) scan += y;
        }
        if (lane == 31) warp_sum[warp] = scan;
        __syncthreads();
        int before_me = scan - sum;
#pragma unroll
        for (int w = 0; w < kCellThreads / 32 - 1; ++w) before_me += w < warp ? warp_sum[w] : 0;
#pragma unroll
        for (int u = 0; u < kOwn; ++u) {  // from marks to moves; kDropped for a member that has left
            int& m = marks.mark[spread(kOwn * threadIdx.x + u)];
            const int mark = m;
            before_me += mark & (kDropped - 1);
            m = mark < kDropped ? (before_me & (kDropped - 1)) - (before_me >> 16) : kDropped;
            before_me += mark & ~(kDropped - 1);
        }
        __syncthreads();
        double2 z[kOwn];
#pragma unroll
        for (int u = 0; u < kOwn; ++u) z[u] = old_values[min(base + kCellThreads * u + int(threadIdx.x), max(nc, 1) - 1)];
#pragma unroll
        for (int u = 0; u < kOwn; ++u) {
            const int k = kCellThreads * u + int(threadIdx.x), move = marks.mark[spread(k)];
            if (k < len && move != kDropped) {
                const int to = base + k + a0 - g0 + move;
                now[to] = marks.member[spread(k)];
                now_values[to] = z[u];
            }
        }
        a0 = a1;
        g0 = g1;
    }
    __syncthreads();
    const double sum = cell_sum<kCellThreads / 32 - 1>(stage, now_values, 0, count);
    if (threadIdx.x < 2) {
        const double was = threadIdx.x ? before.y : before.x;
        const double m = count > 0 ? sum / double(count) : was;
        reinterpret_cast<double*>(codebook_next)[2 * c + threadIdx.x] = m;
        reinterpret_cast<float*>(codebook32_next)[2 * c + threadIdx.x] = float(m);
        const float step = fabsf(float(m - was)) * (1.f + 1e-6f);
        const float other = __shfl_xor_sync(0x3u, step, 1);
        if (threadIdx.x == 0) {
            const unsigned moved = __float_as_uint(sqrtf(step * step + other * other) * (1.f + 1e-6f));
            if (moved > *const_cast<volatile unsigned*>(&state->moved[slot])) atomicMax(&state->moved[slot], moved);
            inc.size[c] = count;
            inc.which[c] = (unsigned char)(which ^ 1);
            inc.n_arrived[c] = inc.n_left[c] = 0;
        }
    }
}

// Initial codewords sqrt(2) * sample_i, and the f32 copy of the codebook that the filter reads.
__global__ void init_kernel(const double2* samples, int K, double2* codebook, float2* codebook32, TrainState* state) {
    chain_release();
    chain_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c == 0) *state = TrainState{};
    if (c >= K) return;
    const double root2 = 1.4142135623730950488016887242097;
    const double2 z = samples[c];
    codebook[c] = make_double2(root2 * z.x, root2 * z.y);
    codebook32[c] = make_float2(float(root2 * z.x), float(root2 * z.y));
}

// Where the scratch memory of a call comes from: a pool per device that keeps up to 256 MB between calls until
// qamw_release_scratch gives them back.  NULL if the device has no pools of its own, or, without `create`, if there is
// none yet.  256 MB are passes in full on 6 million samples; incremental updates on as many take 600, and a call that makes them and
// needs more than 256 raises the limit to 640.  What a call takes from the driver and gives back costs it time: K = 2048, 100
// updates, 3, 4 and 6 million samples 13.6, 18.3 and 28.7 ms with 256 MB kept, 12.7, 16.2 and 24.1 with all (quiet host; up to 0.8 s a
// call where others keep the driver busy).  Beyond that incremental updates still win (8 million: 35.5 against 52.7 in full).
constexpr int kMaxDevices = 64;
constexpr size_t kKeepBytes = size_t(256) << 20, kKeepMore = size_t(640) << 20;
void keep_at_most(cudaMemPool_t pool, uint64_t bytes) { cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &bytes); }
cudaMemPool_t scratch_pool(bool create) {
    static std::mutex mu;
    static cudaMemPool_t pools[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[dev] && create) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        keep_at_most(p, kKeepBytes);
        pools[dev] = p;
    }
    return pools[dev];
}

}  // namespace

extern "C" int qamw_release_scratch(void) {
    cudaMemPool_t pool = scratch_pool(false);
    if (!pool) return QAMW_OK;
    keep_at_most(pool, kKeepBytes);
    cudaError_t e = cudaStreamSynchronize(nullptr);  // the last call's scratch is freed in the order of this stream
    if (e == cudaSuccess) e = cudaMemPoolTrimTo(pool, 0);
    if (e != cudaSuccess) {
        set_cuda_error("qamw_release_scratch", int(e));
        return QAMW_ERR_CUDA;
    }
    return QAMW_OK;
}

extern "C" int qamw_train_codebook_gpu(int K, uint64_t n_samples, uint64_t seed, const double* samples_dev,
                                       int max_iters, double rel_tol, float* codebook_out, double* train_mse_out,
                                       int* iters_out, double* mse_trace_out, double* seconds_out) {
    if (!codebook_out) return QAMW_ERR_ARG;
    if (K < 1 || K > QAMW_MAX_K || !is_pow2(K)) return QAMW_ERR_SHAPE;
    if (n_samples < uint64_t(K) || n_samples >= (uint64_t(1) << 31) || max_iters < 0 || !(rel_tol >= 0.0)) return QAMW_ERR_ARG;
    const auto t_begin = std::chrono::steady_clock::now();
    const unsigned long long n = n_samples;
    const int chunk = std::min(kMaxChunk, std::max(kMinChunk, int(((n + kManyChunks - 1) / kManyChunks + 31) / 32 * 32)));
    const int n_chunks = int((n + chunk - 1) / chunk), n_tiles = int((n + kTile - 1) / kTile);
    const int bins = std::max(K, 256);
    // One allocation, cut into pieces.  Incremental updates need about twice as much again: where that much is not to be had the
    // passes in full remain, which give the same bits.
    bool incremental = K >= kIncrementalK && n / K <= 1024 + 2 * unsigned(K) && max_iters >= kFullFirst;
    const int room = 64 + int(n / unsigned(K) / 4);
    size_t bytes, slots, o_gen, o_sorted, o_cell, o_values, o_ids, o_assign, o_hist, o_start, o_cb, o_cb32, o_err, o_box, o_state, o_scale;
    size_t o_cur, o_near, o_near_n, o_gap, o_members, o_cells, o_changes;
    auto lay_out = [&]() {
        bytes = 0;
        auto piece = [&](size_t b) {
            const size_t at = bytes;
            bytes += (b + 255) & ~size_t(255);
            return at;
        };
        slots = incremental ? n + n / 4 + size_t(room) * (size_t(K) + 1) : 0;
        const size_t tiles = incremental ? size_t(n_tiles) : 0, cells = incremental ? size_t(K) : 0;
        o_gen = piece(samples_dev ? 0 : sizeof(double2) * n);
        o_sorted = piece(sizeof(double2) * n);
        o_cell = piece(sizeof(double2) * std::max<size_t>(n, slots));
        o_values = piece(sizeof(double2) * slots);
        o_ids = piece(sizeof(int) * n);
        o_assign = piece(sizeof(int) * n);
        o_hist = piece(sizeof(int) * size_t(bins) * n_chunks);
        o_start = piece(sizeof(int) * (size_t(bins) + 1));
        o_cb = piece(2 * sizeof(double2) * K);
        o_cb32 = piece(2 * sizeof(float2) * K);
        o_err = piece(sizeof(double) * n_tiles);
        o_box = piece(sizeof(TileBox) * n_tiles * kBoxes);
        o_state = piece(sizeof(TrainState));
        o_scale = piece(sizeof(float));
        o_cur = piece(2 * (incremental ? n : 0));
        o_near = piece(2 * tiles * kNearMost);
        o_near_n = piece(4 * tiles);
        o_gap = piece(4 * tiles);
        o_members = piece(4 * 2 * slots);
        o_cells = piece(4 * (7 * cells + 1));
        o_changes = piece(4 * 2 * cells * kChanges);
    };
    unsigned char* base = nullptr;
    const cudaMemPool_t pool = scratch_pool(true);
    auto take = [&]() {
        lay_out();
        void** const to = reinterpret_cast<void**>(&base);
        return pool ? cudaMallocFromPoolAsync(to, bytes, pool, nullptr) : cudaMallocAsync(to, bytes, nullptr);
    };
    cudaError_t e = take();
    if (e == cudaErrorMemoryAllocation && incremental) {
        cudaGetLastError();
        incremental = false;
        e = take();
    }
    if (e != cudaSuccess) {
        set_cuda_error("qamw_train_codebook_gpu: cudaMallocAsync", int(e));
        return QAMW_ERR_CUDA;
    }
    if (pool && incremental && bytes > kKeepBytes) keep_at_most(pool, kKeepMore);
    struct Free {
        void* p;
        size_t bytes;
        ~Free() {
            cudaFreeAsync(p, nullptr);
            if (bytes > kKeepBytes) cudaStreamSynchronize(nullptr);  // a pool lets go of what it may not keep when it is waited for
        }
    } owner{base, bytes};
    auto ok = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        return e == cudaSuccess;
    };
    double2* generated = reinterpret_cast<double2*>(base + o_gen);
    double2 *sorted = reinterpret_cast<double2*>(base + o_sorted), *by_cell = reinterpret_cast<double2*>(base + o_cell);
    int *ids = reinterpret_cast<int*>(base + o_ids), *assign = reinterpret_cast<int*>(base + o_assign);
    int *hist = reinterpret_cast<int*>(base + o_hist), *start = reinterpret_cast<int*>(base + o_start);
    // two copies of the codebook: an incremental update reads one and writes the other
    double2 *cbs = reinterpret_cast<double2*>(base + o_cb), *d_cb = cbs;
    float2 *cbs32 = reinterpret_cast<float2*>(base + o_cb32), *d_cb32 = cbs32;
    Increments inc{};
    if (incremental) {
        inc.cur = reinterpret_cast<unsigned short*>(base + o_cur);
        inc.near = reinterpret_cast<unsigned short*>(base + o_near);
        inc.near_n = reinterpret_cast<int*>(base + o_near_n);
        inc.near_gap = reinterpret_cast<float*>(base + o_gap);
        inc.members[0] = reinterpret_cast<int*>(base + o_members);
        inc.members[1] = inc.members[0] + slots;
        inc.values[0] = reinterpret_cast<double2*>(base + o_values);
        inc.values[1] = by_cell;  // the full pass's samples by cell, until they are adopted
        inc.size = reinterpret_cast<int*>(base + o_cells);
        inc.slab = inc.size + K;
        inc.n_arrived = inc.slab + K + 1;
        inc.n_left = inc.n_arrived + K;
        inc.order = inc.n_left + K;
        inc.which = reinterpret_cast<unsigned char*>(inc.order + K);
        inc.arrived = reinterpret_cast<int*>(base + o_changes);
        inc.left = inc.arrived + size_t(K) * kChanges;
    }
    double* tile_err = reinterpret_cast<double*>(base + o_err);
    TileBox* boxes = reinterpret_cast<TileBox*>(base + o_box);
    TrainState* state = reinterpret_cast<TrainState*>(base + o_state);
    float* scale = reinterpret_cast<float*>(base + o_scale);
    const double2* samples = samples_dev ? reinterpret_cast<const double2*>(samples_dev) : generated;
    // The kernels run on the default stream; the caller's samples may still be on their way on one that does not wait
    // for it and that it does not wait for.
    if (samples_dev) ok(cudaDeviceSynchronize());
    if (!samples_dev) {
        ok(launch_chained(sample_kernel, 8 * sm_count(), 256, 0, nullptr, sample_key(seed), n, generated));
    }
    auto sort_smem = [](int b) { return sizeof(int) * size_t(b) + size_t(kSortWarps) * size_t((b + 1) & ~1) * 2; };
    if (sort_smem(bins) > 48 * 1024)  // beyond the default dynamic limit
        ok(cudaFuncSetAttribute(scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sort_smem(bins))));
    ok(launch_chained(init_kernel, (K + 255) / 256, 256, 0, nullptr, samples, K, d_cb, d_cb32, state));

    // spatial order: two stable passes over the Hilbert position's bytes (the cells' buffers are free so far)
    int *pos = assign, *half = reinterpret_cast<int*>(by_cell);
    ok(launch_chained(scale_kernel, 1, 1024, 0, nullptr, samples, n, scale));
    ok(launch_chained(hilbert_kernel, 8 * sm_count(), 256, 0, nullptr, samples, n, scale, pos));
    for (int pass = 0; pass < 2; ++pass) {
        const KeyOf key{pos, pass ? half : nullptr, 8 * pass, 255};
        ok(launch_chained(hist_kernel, n_chunks, 512, sizeof(int) * 256, nullptr, key, n, chunk, 256, hist, nullptr, 0, 0.0, 0, state));
        ok(launch_chained(prefix_kernel, 8, 1024, 0, nullptr, hist, n_chunks, 256, start, state));
        ok(launch_chained(scatter_kernel, n_chunks, 32 * kSortWarps, sort_smem(256), nullptr, key, n, chunk, 256, hist, start, samples, pass ? ids : half,
                                                            pass ? sorted : nullptr, nullptr));
    }
    ok(launch_chained(box_kernel, n_tiles, kTile, 0, nullptr, sorted, n, boxes));

    auto assign_pass = [&](int* to, const TrainState* st) {
        auto go = [&](auto kernel) {
            ok(launch_chained(kernel, n_tiles, kTile, 0, nullptr, sorted, ids, n, boxes, d_cb, d_cb32, K, to, tile_err, st));
        };
        switch (K / kTile) {
            case 16: go(assign_kernel<16>); break;
            case 8: go(assign_kernel<8>); break;
            case 4: go(assign_kernel<4>); break;
            case 2: go(assign_kernel<2>); break;
            default: go(assign_kernel<1>); break;
        }
    };
    const KeyOf cell{assign, nullptr, 0, 0x7fffffff};
    auto full_pass = [&](int* ids_out) {
        assign_pass(assign, state);
        ok(launch_chained(hist_kernel, n_chunks + 1, kRuleThreads, sizeof(int) * K, nullptr, cell, n, chunk, K, hist, tile_err, n_tiles, rel_tol,
                          max_iters, state));
        ok(launch_chained(prefix_kernel, (K + 31) / 32, 1024, 0, nullptr, hist, n_chunks, K, start, state));
        ok(launch_chained(scatter_kernel, n_chunks, 32 * kSortWarps, sort_smem(K), nullptr, cell, n, chunk, K, hist, start, samples, ids_out,
                          by_cell, state));
        ok(launch_chained(centroid_kernel, K, 64, 0, nullptr, by_cell, start, d_cb, d_cb32, state));
    };
    auto list_near = [&](const int* from) {
        auto go = [&](auto kernel) { ok(launch_chained(kernel, n_tiles, kTile, 0, nullptr, ids, n, boxes, d_cb32, K, from, inc, state)); };
        switch (K / kTile) {
            case 16: go(near_kernel<16>); break;
            case 8: go(near_kernel<8>); break;
            case 4: go(near_kernel<4>); break;
            case 2: go(near_kernel<2>); break;
            default: go(near_kernel<1>); break;
        }
    };
    TrainState seen{};
    int recorded = 0, full_left = kFullFirst, since_near = 0;
    while (e == cudaSuccess) {
        const int updates_before = seen.updates;
        const double2* const cb_before = d_cb;
        int full = 0;
        for (int k = 0; k < kBatch && recorded + k <= max_iters; ++k) {
            if (!incremental || full_left > 0) {
                const bool last = incremental && --full_left == 0;
                full_pass(last ? inc.members[1] : nullptr);
                ++full;
                if (last) {
                    ok(launch_chained(adopt_kernel, K, 256, 0, nullptr, inc.members[1], by_cell, start, room, inc, state));
                    list_near(assign);
                    since_near = 0;
                }
                continue;
            }
            if (since_near == (recorded + k < kEarly ? kNearEarly : kNearLate)) {
                list_near(nullptr);
                since_near = 0;
            }
            double2* next = d_cb == cbs ? cbs + K : cbs;
            float2* next32 = d_cb == cbs ? cbs32 + K : cbs32;
            ok(launch_chained(near_assign_kernel, n_tiles, kNearThreads, 0, nullptr, sorted, ids, n, boxes, d_cb, d_cb32, K, inc, tile_err, state));
            ok(launch_chained(update_kernel, K + 1, kCellThreads, 0, nullptr, samples, n, inc, d_cb, next, next32, tile_err, n_tiles, rel_tol,
                              max_iters, since_near, state));
            ++since_near;
            d_cb = next;
            d_cb32 = next32;
        }
        if (!ok(cudaMemcpy(&seen, state, sizeof(seen), cudaMemcpyDeviceToHost))) break;
        for (; recorded < seen.passes; ++recorded)
            if (mse_trace_out) mse_trace_out[recorded] = seen.trace[recorded % kBatch];
        // the copy of the codebook that the last update wrote: incremental ones change sides
        const bool other = std::max(0, seen.updates - updates_before - full) & 1;
        const bool at_first = (cb_before == cbs) != other;
        d_cb = at_first ? cbs : cbs + K;
        d_cb32 = at_first ? cbs32 : cbs32 + K;
        if (seen.done) break;
        if (seen.stalled) {
            ok(cudaMemsetAsync(&state->stalled, 0, 3 * sizeof(int), nullptr));  // and skip and held
            full_left = kFullAgain;
        }
    }
    std::vector<double> cb(size_t(2) * K);
    ok(cudaMemcpy(cb.data(), d_cb, sizeof(double) * 2 * K, cudaMemcpyDeviceToHost));
    if (e != cudaSuccess) {
        set_cuda_error("qamw_train_codebook_gpu", int(e));
        return QAMW_ERR_CUDA;
    }
    // order by (squared radius, angle) so that indices are reproducible, round to f32
    std::vector<int> order(size_t(K), 0);
    for (int k = 0; k < K; ++k) order[size_t(k)] = k;
    auto r2 = [&](int k) { return cb[2 * size_t(k)] * cb[2 * size_t(k)] + cb[2 * size_t(k) + 1] * cb[2 * size_t(k) + 1]; };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        const double ra = r2(a), rb = r2(b);
        if (ra != rb) return ra < rb;
        return std::atan2(cb[2 * size_t(a) + 1], cb[2 * size_t(a)]) < std::atan2(cb[2 * size_t(b) + 1], cb[2 * size_t(b)]);
    });
    for (int k = 0; k < K; ++k) {
        codebook_out[2 * k] = float(cb[2 * size_t(order[size_t(k)])]);
        codebook_out[2 * k + 1] = float(cb[2 * size_t(order[size_t(k)]) + 1]);
    }
    if (train_mse_out) {  // the error of the returned f32 codebook
        for (int c = 0; c < 2 * K; ++c) cb[size_t(c)] = double(codebook_out[c]);
        ok(cudaMemcpy(d_cb, cb.data(), sizeof(double) * 2 * K, cudaMemcpyHostToDevice));
        ok(cudaMemcpy(d_cb32, codebook_out, sizeof(float) * 2 * K, cudaMemcpyHostToDevice));
        assign_pass(nullptr, nullptr);
        std::vector<double> err(size_t(n_tiles), 0.0);
        ok(cudaMemcpy(err.data(), tile_err, sizeof(double) * n_tiles, cudaMemcpyDeviceToHost));
        double total = 0.0;
        for (double v : err) total += v;
        *train_mse_out = total / double(n);
    }
    if (iters_out) *iters_out = seen.updates;
    if (e != cudaSuccess) {
        set_cuda_error("qamw_train_codebook_gpu", int(e));
        return QAMW_ERR_CUDA;
    }
    if (seconds_out) *seconds_out = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_begin).count();
    return QAMW_OK;
}
