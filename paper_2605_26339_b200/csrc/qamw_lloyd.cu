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
// samples: a sample is compared with about 3 of 2048 codewords instead of all.  The filter runs in f32 with its bounds widened by more than f32 rounding; the
// comparison itself is the full double arithmetic, so the result is that of the exhaustive scan.
//
// Centroids.  A stable counting sort by cell (per-chunk histograms, prefix sums, a scatter that ranks
// equal keys inside a warp by lane) brings every cell's samples together in sample order.  The chain
// of additions of a cell is serial by contract; one warp stages its samples in shared memory and two lanes
// add up x and y.
//
// The stopping rule is evaluated on the device: a batch of iterations is enqueued at once, the kernels
// after the last wanted update return at once, and the host reads the errors once per batch.
//
// K = 2048 on 2^20 samples, 100 updates on a B200: 235 ms with the exhaustive scan, a serial scan of the histograms
// and one host round trip per update; 8.6 to 9.2 ms now, by box.
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
constexpr int kBatch = 8;            // iterations enqueued between two looks at the stopping rule

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
    unsigned ticket;         // blocks of the prefix kernel that have finished; zero between launches
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
// are candidates.  One for each warp's 32 samples, and one for the whole tile.
struct TileBox {
    float mx, my, rx, ry;
};
constexpr int kTileWarps = kTile / 32;
constexpr int kBoxes = kTileWarps + 1;  // per tile: the warps', then the tile's
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
    __shared__ int any_bad;
    if (threadIdx.x == 0) any_bad = 0;
    __syncthreads();
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
        if (bad) any_bad = 1;
        boxes[size_t(blockIdx.x) * kBoxes + w] = make_box(x0, x1, y0, y1, bad);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kTileWarps; ++k) {
            x0 = fmin(x0, lo[0][k]);
            x1 = fmax(x1, hi[0][k]);
            y0 = fmin(y0, lo[1][k]);
            y1 = fmax(y1, hi[1][k]);
        }
        boxes[size_t(blockIdx.x) * kBoxes + kTileWarps] = make_box(x0, x1, y0, y1, any_bad != 0);
    }
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

// Exact nearest codeword of the samples of a tile: d = dx*dx + dy*dy with one rounding per
// operation (no fused multiply-add: the result must not depend on how a compiler contracts the
// expression), the lowest index among equal distances.  Also adds up the distances of the tile in a fixed
// order (a shuffle tree, then by warp).  Bound by the f32 filter over all codewords (K / 256 per thread) and
// the waits between its four steps, which is why the SM is filled with small blocks (eight of 256 threads; three of
// 512: 9.06 against 8.93 ms a call at K = 2048, 12.3 against 9.8 at K = 512), then by
// the double comparisons with those that remain; both arrays come from L1/L2.
template <int PER>  // codewords per thread: K / kTile, or 1 for a smaller codebook
__global__ void __launch_bounds__(kTile, 8) assign_kernel(const double2* sorted, const int* ids, unsigned long long n,
                                                       const TileBox* boxes, const double2* codebook,
                                                       const float2* codebook32, int K, int* assign, double* tile_err,
                                                       const TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ unsigned short list[QAMW_MAX_K];
    __shared__ double2 cand[kTile];
    __shared__ float2 cand32[kTile];
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
    double best = INFINITY;
    int arg = 0;
    for (int base = 0; base < count; base += kTile) {
        const int part = min(kTile, count - base);
        if (base) __syncthreads();  // the previous candidates have been read
        if (threadIdx.x < part) {
            const int c = list[base + threadIdx.x];
            cand[threadIdx.x] = codebook[c];
            cand32[threadIdx.x] = codebook32[c];
        }
        __syncthreads();
        // of these, the ones that can be nearest to a point of the warp's own box
        float wf = INFINITY, wn = INFINITY;
        for (int k = lane; k < part; k += 32) {
            float f;
            box_bounds(bw, cand32[k], wn, f);
            wf = fminf(wf, f);
        }
        const float wmin = __uint_as_float(__reduce_min_sync(kFullMask, __float_as_uint(wf)));
        const float wlimit = bw.rx < 0.f ? INFINITY : wmin + kTiny;
        for (int k0 = 0; k0 < part; k0 += 32) {
            float near = wn;  // already there when all fit one step
            if (part > 32 && k0 + lane < part) {
                float f;
                box_bounds(bw, cand32[k0 + lane], near, f);
            }
            unsigned keep = __ballot_sync(kFullMask, k0 + lane < part && !(near > wlimit));
            while (keep) {
                const int k = k0 + __ffs(int(keep)) - 1;
                keep &= keep - 1;
                const double2 q = cand[k];
                const int c = list[base + k];
                const double dx = __dsub_rn(z.x, q.x), dy = __dsub_rn(z.y, q.y);
                const double d = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
                // the list is in no particular order: among equals the lowest index
                arg = d < best ? c : d == best ? min(arg, c) : arg;
                best = d < best ? d : best;
            }
        }
    }
    if (best == INFINITY) arg = 0;  // not a number: as the exhaustive scan, which starts from codeword 0
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

// Histogram of one chunk: hist[chunk * bins + bin].  In a training pass one more block adds up the tiles'
// errors in a fixed order and applies the stopping rule, beside the others.
__global__ void __launch_bounds__(512) hist_kernel(KeyOf key, unsigned long long n, int chunk, int bins, int* hist,
                                                   const double* tile_err, int n_tiles, double rel_tol, int max_iters,
                                                   TrainState* state) {
    chain_release();
    chain_wait();
    extern __shared__ int h[];
    __shared__ double err_part[16];
    if (tile_err && state->done) return;
    const unsigned long long lo = blockIdx.x * (unsigned long long)chunk, hi = min(n, lo + chunk);
    if (lo >= n) {
        double e = 0.0;
        for (int i = threadIdx.x; i < n_tiles; i += 512) e += tile_err[i];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) e += __shfl_xor_sync(kFullMask, e, s);
        if ((threadIdx.x & 31) == 0) err_part[threadIdx.x >> 5] = e;
        __syncthreads();
        if (threadIdx.x == 0) {
            double total = 0.0;
            for (int w = 0; w < 16; ++w) total += err_part[w];
            const double D = total / double(n);
            state->trace[state->passes++ % kBatch] = D;
            if ((state->passes > 1 && state->prev - D <= rel_tol * state->prev) || state->updates >= max_iters)
                state->done = 1;
            else
                ++state->updates;
            state->prev = D;
        }
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

// New codewords: a warp adds the samples of one cell in sample order and divides by their number; an
// empty cell keeps its codeword.  The additions are one serial chain per coordinate (lane 0: x, lane 1:
// y); the other lanes keep the next 64 samples coming and the two lanes read theirs sixteen ahead.  The pass lasts as
// long as the chain of its largest cell, at 11 to 12 clocks an addition, of which a dependent addition in registers
// takes 8.  A trained codebook's largest cells, at the centre, hold twice the mean, 2 n / K: 2^20 samples take 14 us an
// update at K = 2048, 200 us at K = 64 and 3 ms at K = 2, where a call (100 updates) takes 8.8, 27 and 300 ms.  The
// order of the additions is part of the result, so only the 3 to 4 clocks beside the addition could be saved.
constexpr int kCellWarps = 4;
__global__ void __launch_bounds__(32 * kCellWarps) centroid_kernel(const double2* by_cell, const int* start, int K,
                                                                   double2* codebook, float2* codebook32,
                                                                   const TrainState* state) {
    chain_release();
    chain_wait();
    __shared__ __align__(16) double stage[kCellWarps][2][CellWalk::kStep];
    if (state->done) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * kCellWarps + warp;
    if (c >= K) return;
    const int lo = start[c], hi = start[c + 1];
    if (hi <= lo) return;
    double (*st)[64] = stage[warp];
    CellWalk walk(lo, hi);
    auto sample = [&](int k) { return walk.has(k) ? by_cell[walk.at(k)] : make_double2(0.0, 0.0); };
    double2 a = sample(lane), b = sample(32 + lane);
    double sum = 0.0;
    for (; walk.more(); walk.step()) {
        st[0][lane] = a.x;
        st[1][lane] = a.y;
        st[0][32 + lane] = b.x;
        st[1][32 + lane] = b.y;
        a = sample(64 + lane);
        b = sample(96 + lane);
        __syncwarp();
        if (lane < 2) {
            if (walk.full()) {
                const double2* v = reinterpret_cast<const double2*>(st[lane]);
                double2 q[2][8];
#pragma unroll
                for (int k = 0; k < 8; ++k) q[0][k] = v[k];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    if (g < 3) {
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
                for (int k = 0; k < walk.left(); ++k) sum += st[lane][k];
            }
        }
        __syncwarp();
    }
    if (lane < 2) {
        const double m = sum / double(hi - lo);
        reinterpret_cast<double*>(codebook)[2 * c + lane] = m;
        reinterpret_cast<float*>(codebook32)[2 * c + lane] = float(m);
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

// Where the scratch memory of a call comes from: a pool per device that keeps up to 256 MB between calls (the
// default size takes 60 MB; with cudaMalloc and cudaFree a call cost 3 ms more) until qamw_release_scratch gives it
// back.  NULL if the device has no pools of its own, or, without `create`, if there is none yet.
constexpr int kMaxDevices = 64;
constexpr size_t kKeepBytes = size_t(256) << 20;
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
        uint64_t keep = kKeepBytes;
        cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        pools[dev] = p;
    }
    return pools[dev];
}

}  // namespace

extern "C" int qamw_release_scratch(void) {
    cudaMemPool_t pool = scratch_pool(false);
    if (!pool) return QAMW_OK;
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
    // one allocation, cut into pieces
    size_t bytes = 0;
    auto piece = [&](size_t b) {
        const size_t at = bytes;
        bytes += (b + 255) & ~size_t(255);
        return at;
    };
    const size_t o_gen = piece(samples_dev ? 0 : sizeof(double2) * n), o_sorted = piece(sizeof(double2) * n),
                 o_cell = piece(sizeof(double2) * n), o_ids = piece(sizeof(int) * n), o_assign = piece(sizeof(int) * n),
                 o_hist = piece(sizeof(int) * size_t(bins) * n_chunks), o_start = piece(sizeof(int) * (size_t(bins) + 1)),
                 o_cb = piece(sizeof(double2) * K), o_cb32 = piece(sizeof(float2) * K), o_err = piece(sizeof(double) * n_tiles),
                 o_box = piece(sizeof(TileBox) * n_tiles * kBoxes), o_state = piece(sizeof(TrainState)), o_scale = piece(sizeof(float));
    unsigned char* base = nullptr;
    cudaError_t e = cudaSuccess;
    if (cudaMemPool_t pool = scratch_pool(true)) {
        e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&base), bytes, pool, nullptr);
    } else {
        e = cudaMallocAsync(reinterpret_cast<void**>(&base), bytes, nullptr);
    }
    if (e != cudaSuccess) {
        set_cuda_error("qamw_train_codebook_gpu: cudaMallocAsync", int(e));
        return QAMW_ERR_CUDA;
    }
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
    double2* d_cb = reinterpret_cast<double2*>(base + o_cb);
    float2* d_cb32 = reinterpret_cast<float2*>(base + o_cb32);
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
    TrainState seen{};
    int recorded = 0;
    while (e == cudaSuccess) {
        for (int k = 0; k < kBatch && recorded + k <= max_iters; ++k) {
            assign_pass(assign, state);
            ok(launch_chained(hist_kernel, n_chunks + 1, 512, sizeof(int) * K, nullptr, cell, n, chunk, K, hist, tile_err, n_tiles, rel_tol, max_iters,
                                                                 state));
            ok(launch_chained(prefix_kernel, (K + 31) / 32, 1024, 0, nullptr, hist, n_chunks, K, start, state));
            ok(launch_chained(scatter_kernel, n_chunks, 32 * kSortWarps, sort_smem(K), nullptr, cell, n, chunk, K, hist, start, samples, nullptr, by_cell, state));
            ok(launch_chained(centroid_kernel, (K + kCellWarps - 1) / kCellWarps, 32 * kCellWarps, 0, nullptr, by_cell, start, K, d_cb, d_cb32, state));
        }
        if (!ok(cudaMemcpy(&seen, state, sizeof(seen), cudaMemcpyDeviceToHost))) break;
        for (; recorded < seen.passes; ++recorded)
            if (mse_trace_out) mse_trace_out[recorded] = seen.trace[recorded % kBatch];
        if (seen.done) break;
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
