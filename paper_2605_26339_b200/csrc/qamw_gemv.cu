// Fused decode -> matrix-vector product: y = W_hat x straight from the packed stream, without ever
// writing W_hat (the paper's pipeline dequantises to BF16 before the matmul and names the fused kernel
// as its main engineering follow-up: Section 1, Limitations).
//
// Row i of the decoder's output is  w_hat_i = r_i D_s^-1 S F yhat_i  (Section 3.2, B.2), with
// yhat_i = (sigma_k c_idx_k)_k the scaled codewords and F the symmetric, orthonormal block Hadamard
// matrix (Lemma 1).  Hence
//     w_hat_i . x  =  r_i  yhat_i . (F S D_s^-1 x)  =  r_i  sum_k  c_idx_k . (sigma_k xt_k),
// where xt = R_fwd (x / s) is the *activation* rotated once per call.  The per-row inverse rotation
// disappears: a row costs one codeword gather and two fused multiply-adds per pair, and reads B/16
// bytes per weight instead of the 2 bytes of a BF16 matrix.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <unordered_map>

#include "qamw_device.cuh"
#include "qamw_internal.h"
#include "qamw_launch.h"

using namespace qamw;

namespace {

// xt = F S (x / s), pair k scaled by sigma_k, for one activation vector per block; written chunk-
// transposed: pair 16 c + i of vector v at out[(v * 16 + i) * n_chunks + c], so that the lanes of the
// product kernel (one chunk of 16 pairs each) read consecutive addresses.
__global__ void gemv_rotate_kernel(const float* x, const float* chan_scale, const int8_t* signs, const float* sigma,
                                   int d_in, int log2b, float2* out) {
    extern __shared__ float v[];
    chain_release();
    chain_wait();
    const int vec = blockIdx.x;
    const float* xv = x + size_t(vec) * d_in;
    for (int j = threadIdx.x; j < d_in; j += blockDim.x)
        v[j] = float(signs[j]) * xv[j] / (chan_scale ? chan_scale[j] : 1.0f);
    __syncthreads();
    for (int s = 0; s < log2b; ++s) {  // butterflies of every block, stage h = 2^s
        const int h = 1 << s;
        for (int t = threadIdx.x; t < d_in / 2; t += blockDim.x) {
            const int lo = ((t >> s) << (s + 1)) | (t & (h - 1));
            const float a = v[lo], c = v[lo + h];
            v[lo] = a + c;
            v[lo + h] = a - c;
        }
        __syncthreads();
    }
    const float scale = rsqrtf(float(1 << log2b));
    const int n_pairs = d_in >> 1, n_chunks = n_pairs >> 4;
    for (int k = threadIdx.x; k < n_pairs; k += blockDim.x) {
        const float sg = sigma[k] * scale;
        out[(size_t(vec) * 16 + (k & 15)) * n_chunks + (k >> 4)] = make_float2(v[2 * k] * sg, v[2 * k + 1] * sg);
    }
}

struct GemvArgs {
    const uint8_t* packed;
    long long stride;
    const float* row_norm;
    const float2* codebook;
    const float2* xt;  // rotated activations, chunk-transposed (see gemv_rotate_kernel)
    float* y;
    int d_out, n_pairs, K, B, log2c;
};

// One warp per row at a time, a lane per chunk of 16 pairs: 16 B index bits read as 32-bit words
// (rows are 4-byte aligned), cut with funnel shifts, codewords from bank-separated copies in shared
// memory, the rotated activations of all vectors from shared memory too.
template <int NVEC>
__global__ void __launch_bounds__(512, 1) gemv_kernel(const GemvArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int B = a.B;
    const uint32_t mask = (1u << B) - 1u;
    const uint32_t cb_stride = 8u << a.log2c;
    const uint32_t cb = smem_addr(smem) + 8u * (threadIdx.x & ((1 << a.log2c) - 1));
    const int n_chunks = a.n_pairs >> 4;
    float2* xs = reinterpret_cast<float2*>(smem + ((size_t(a.K) * 8) << a.log2c));
    chain_release();
    fill_codebook_copies(reinterpret_cast<float2*>(smem), a.codebook, a.K, a.log2c);
    chain_wait();
    for (int i = threadIdx.x; i < NVEC * 16 * n_chunks; i += blockDim.x) xs[i] = a.xt[i];
    __syncthreads();
    const int words_per_chunk = B / 2;          // 16 B bits = B / 2 words when B is even ...
    const int row_words = int((((long long)a.n_pairs * B + 7) / 8 + 3) / 4);
    for (int row = blockIdx.x * n_warps + warp; row < a.d_out; row += gridDim.x * n_warps) {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(a.packed + (long long)row * a.stride);
        float acc[NVEC];
#pragma unroll
        for (int v = 0; v < NVEC; ++v) acc[v] = 0.f;
        for (int c = lane; c < n_chunks; c += 32) {
            // ... and in general the chunk starts at bit 16 B c: word (B c) / 2, shift 16 (B c & 1)
            const unsigned bit0 = 16u * unsigned(B) * unsigned(c);
            const int w0 = int(bit0 >> 5);
            const uint32_t sh = bit0 & 31u;
            uint32_t word[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) word[i] = (i <= words_per_chunk + 1 && w0 + i < row_words) ? w[w0 + i] : 0u;
            // shift the window down to bit 0, then cut two indices per step of 2 B bits
            uint32_t win[7];
#pragma unroll
            for (int i = 0; i < 7; ++i) win[i] = __funnelshift_r(word[i], word[i + 1], sh);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const uint32_t i0 = win[0] & mask, i1 = (win[0] >> B) & mask;
                const float2 c0 = lds_f32x2(cb + i0 * cb_stride), c1 = lds_f32x2(cb + i1 * cb_stride);
#pragma unroll
                for (int v = 0; v < NVEC; ++v) {
                    const float2 x0 = xs[(v * 16 + 2 * t) * n_chunks + c], x1 = xs[(v * 16 + 2 * t + 1) * n_chunks + c];
                    acc[v] = fmaf(c0.x, x0.x, acc[v]);
                    acc[v] = fmaf(c0.y, x0.y, acc[v]);
                    acc[v] = fmaf(c1.x, x1.x, acc[v]);
                    acc[v] = fmaf(c1.y, x1.y, acc[v]);
                }
                if (t < 7) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) win[i] = __funnelshift_r(win[i], win[i + 1], 2 * B);
                    win[6] >>= 2 * B;
                }
            }
        }
        const float rn = a.row_norm[row];
#pragma unroll
        for (int v = 0; v < NVEC; ++v) {
            float s = acc[v];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
            if (lane == 0) a.y[size_t(row) * NVEC + v] = rn * s;
        }
    }
}

__device__ __forceinline__ uint32_t lds_word(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// ---------------------------------------------------------------------------------------------
// Fast path: column slices in registers.
//
// Block b owns rows b, b + gridDim, b + 2 gridDim, ...  Its warps form G row groups of S_par warps; a
// warp owns one *slice* of 512 pairs (1024 columns) and walks every G-th row of the block, two at a time.
// Lane l holds the rotated, scaled activations of chunk 32 slice + l (16 pairs, 32 floats per vector) in
// registers -- a slice is a whole number of Hadamard blocks, so a warp can rotate its own -- and a
// pair costs one codeword gather and one packed fused multiply-add per vector.  The 64 B bytes of a
// row's slice arrive through a ring of 16-byte asynchronous copies, several rows ahead; a row that starts off
// a 16-byte boundary is copied from the boundary below it and read at an offset.  The slices'
// partial sums of a tile of rows meet in shared memory behind one block barrier per tile and are
// added in ascending slice order, so the result does not depend on timing.  Rows longer than the
// block has warps for are walked in several passes, each adding into y.
//
// Bound by the shared-memory pipe: a gather of 32 codewords takes 4 wavefronts from eight copies (K = 2048), the
// index words 0.75, copies, sums and staging 1, which is 20 us for the 35.4 M pairs of 13824 x 5120 on 148 SMs.  The
// width B of an index is a template parameter for the bitrates in use, so that every index is cut out at a fixed
// position, and the two rows of a step share the activations, which keeps 32 gathers in flight with the few warps
// that 32 registers per vector leave room for.
// ---------------------------------------------------------------------------------------------
struct Gemv2Args {
    const uint8_t* packed;
    long long stride;
    const float* x;           // [n_vec, d_in]
    const float* chan_scale;  // or NULL
    const int8_t* signs;
    const float* sigma;
    const float2* codebook;
    const float* row_norm;
    float4* xt;               // four vectors: rotated activations, see xt_index
    float* y;                 // [d_out][n_vec]
    int d_out, d_in, n_chunks, n_slices, K, B, log2c, log2b;
    int s_par;                // slices walked side by side: ceil(n_slices / passes)
    int seg_bytes, stage_bytes;
    float inv_sqrt_b;
};

template <int NVEC>
struct GemvGeom {
    static constexpr int kThreads = NVEC == 4 ? 320 : NVEC == 2 ? 384 : 512;  // 32 activation registers per thread and vector; warps per scheduler set the register cap
    static constexpr int kDepth = 6;       // staged rows per warp, in pairs: about 40 KB in flight per SM
    static constexpr int kTileRows = 32;   // rows per warp between two block barriers
};
constexpr int kRotateStage = 32 * 144;     // shared memory of rotate_slice: 32 chunks of 128 bytes, 16 apart

// Sums of N per-lane values over the warp: while more than one value is left, a step halves the number that a lane
// carries.  Afterwards the lanes with (lane & (32 / N - 1)) == 0 hold value lane / (32 / N).
template <int N>
__device__ __forceinline__ float warp_sums(float (&v)[N], int lane) {
    int m = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n /= 2, m /= 2) {
        const bool up = lane & m;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
            v[i] = keep + __shfl_xor_sync(kFull, send, m);
        }
    }
    for (; m >= 1; m /= 2) v[0] += __shfl_xor_sync(kFull, v[0], m);
    return v[0];
}


// Rotated activations of one slice, by one warp: lane l gets chunk 32 slice + l of each vector,
// xr[v][i] = sigma_k (F S D_s^-1 x_v) at pair k = 16 chunk + i; zero beyond the row.  The columns are read
// lane by lane along the row and handed to their chunks through `stage` (read at a chunk per lane they
// took 32 wavefronts a load and 5 of the 30 us of 13824 x 5120).
template <int NVEC>
__device__ __forceinline__ void rotate_slice(const Gemv2Args& a, int slice, int v0, unsigned char* stage, int lane, f32x2 (&xr)[NVEC][16]) {
    const int col0 = 1024 * slice, chunk = 32 * slice + lane;
    // the loads of a vector before the first store to `stage`, which the compiler must take for a store to `x`
    float4 q[8];
    auto fetch = [&](int v) {
        const float* x = a.x + size_t(v0 + v) * a.d_in;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int col = col0 + 128 * e + 4 * lane;
            q[e] = col < a.d_in ? *reinterpret_cast<const float4*>(x + col) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    fetch(0);
    float4 sg4[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
        sg4[e] = chunk < a.n_chunks ? reinterpret_cast<const float4*>(a.sigma + 16 * chunk)[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    float tj[32];  // sign_j / s_j of columns col0 + 128 e + 4 lane + i
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int col = col0 + 128 * e + 4 * lane;
        const bool in = col < a.d_in;
        const uint32_t sw = in ? *reinterpret_cast<const uint32_t*>(a.signs + col) : 0u;
        float4 s = make_float4(1.f, 1.f, 1.f, 1.f);
        if (in && a.chan_scale) s = *reinterpret_cast<const float4*>(a.chan_scale + col);
        tj[4 * e] = __fdividef(float(int(int8_t(sw & 0xffu))), s.x);
        tj[4 * e + 1] = __fdividef(float(int(int8_t((sw >> 8) & 0xffu))), s.y);
        tj[4 * e + 2] = __fdividef(float(int(int8_t((sw >> 16) & 0xffu))), s.z);
        tj[4 * e + 3] = __fdividef(float(int(int8_t(sw >> 24))), s.w);
    }
#pragma unroll
    for (int v = 0; v < NVEC; ++v) {
        __syncwarp();  // the staging memory is free
#pragma unroll
        for (int e = 0; e < 8; ++e)
            *reinterpret_cast<float4*>(stage + (4 * e + (lane >> 3)) * 144 + (lane & 7) * 16) =
                make_float4(q[e].x * tj[4 * e], q[e].y * tj[4 * e + 1], q[e].z * tj[4 * e + 2], q[e].w * tj[4 * e + 3]);
        if (v + 1 < NVEC) fetch(v + 1);
        __syncwarp();
        float t[32];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float4 u = *reinterpret_cast<const float4*>(stage + lane * 144 + 16 * e);
            t[4 * e] = u.x;
            t[4 * e + 1] = u.y;
            t[4 * e + 2] = u.z;
            t[4 * e + 3] = u.w;
        }
#pragma unroll
        for (int st = 0; st < 5; ++st) {  // butterflies inside the lane's 32 columns
            if (st < a.log2b) {
                const int h = 1 << st;
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (!(e & h)) {
                        const float lo = t[e], up = t[e + h];
                        t[e] = lo + up;
                        t[e + h] = lo - up;
                    }
            }
        }
        for (int st = 5; st < a.log2b; ++st) {  // blocks wider than a chunk: lanes 2^(st-5) apart
            const int m = 1 << (st - 5);
            const bool upper = lane & m;
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const float o = __shfl_xor_sync(kFull, t[e], m);
                t[e] = upper ? o - t[e] : t[e] + o;
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float sg[4] = {sg4[e].x * a.inv_sqrt_b, sg4[e].y * a.inv_sqrt_b, sg4[e].z * a.inv_sqrt_b, sg4[e].w * a.inv_sqrt_b};
#pragma unroll
            for (int i = 0; i < 4; ++i) xr[v][4 * e + i] = pack2(t[8 * e + 2 * i] * sg[i], t[8 * e + 2 * i + 1] * sg[i]);
        }
    }
    __syncwarp();
}

// Where the rotated activations of four vectors lie: by slice, vector and group of two pairs, one float4 per live
// lane, so that a warp reads whole lines and the whole takes no more than the vectors themselves.
__device__ __forceinline__ size_t xt_index(const Gemv2Args& a, int slice, int v, int j, int lane) {
    return size_t(slice) * 1024 + (v * 8 + j) * min(32, a.n_chunks - 32 * slice) + lane;
}
constexpr int kRotateWarps = 4;
__global__ void __launch_bounds__(32 * kRotateWarps) gemv_rotate4_kernel(const Gemv2Args a) {
    __shared__ __align__(16) unsigned char stage[kRotateWarps][kRotateStage];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;  // a warp per vector, a block per slice
    chain_release();
    chain_wait();
    f32x2 xr[1][16];
    rotate_slice<1>(a, blockIdx.x, warp, stage[warp], lane, xr);
    if (32 * int(blockIdx.x) + lane >= a.n_chunks) return;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float4 o;
        unpack2(xr[0][2 * j], o.x, o.y);
        unpack2(xr[0][2 * j + 1], o.z, o.w);
        a.xt[xt_index(a, blockIdx.x, warp, j, lane)] = o;
    }
}

// BT: bits of an index, or 0 for the widths below 6, read from the arguments
template <int NVEC, int BT>
__device__ __forceinline__ void gemv2_rows(const Gemv2Args& a) {
    constexpr int R = 2, D = GemvGeom<NVEC>::kDepth;
    constexpr int BMAX = BT ? BT : 5;
    constexpr bool ODD = BT == 0 || BT % 2;                         // a chunk may start in the middle of a word
    constexpr int NB = (16 * BMAX + 31) / 32;                      // words of a lane's 16 indices,
    constexpr int NW = (16 * BMAX + (ODD ? 16 : 0) + 31) / 32;     // and of what they are cut from
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int B = BT ? BT : a.B;
    const uint32_t mask = (1u << B) - 1u;
    const uint32_t cb_stride = 8u << a.log2c;
    const uint32_t cb = smem_addr(smem) + 8u * (threadIdx.x & ((1 << a.log2c) - 1));
    unsigned char* stage = smem + ((size_t(a.K) * 8) << a.log2c) + size_t(warp) * D * a.stage_bytes;
    const uint32_t stage_addr = smem_addr(stage);

    const int S = a.n_slices;
    const int S_par = a.s_par;                // slices walked side by side
    const int G = n_warps / S_par;            // row groups
    const int s0 = warp % S_par, g = warp / S_par;
    constexpr int JT = GemvGeom<NVEC>::kTileRows;
    const int TI = JT * G;                    // rows of the block per tile
    // rows of this block: blockIdx.x + gridDim.x * i, i < n_b
    const int n_b = int(blockIdx.x) < a.d_out ? (a.d_out - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x) : 0;
    const int n_tiles = (n_b + TI - 1) / TI;
    float* ps_base = reinterpret_cast<float*>(smem + ((size_t(a.K) * 8) << a.log2c) + size_t(n_warps) * D * a.stage_bytes);
    // where the lane's 16 B index bits start inside a staged segment
    const uint32_t w_off = 4u * ((uint32_t(B) * uint32_t(lane)) >> 1), sh = ((uint32_t(B) * uint32_t(lane)) & 1u) * 16u;
    const int row_bytes = int((((long long)(a.d_in >> 1)) * B + 7) / 8 + 3) & ~3;  // <= stride (a multiple of 4)
    const long long src_step = (long long)G * int(gridDim.x) * a.stride;

    chain_release();
    fill_codebook_copies(reinterpret_cast<float2*>(smem), a.codebook, a.K, a.log2c);
    chain_wait();
    __syncthreads();

    for (int pass = 0; pass * S_par < S; ++pass) {
        const int slice = pass * S_par + s0;
        const int n_live = min(S_par, S - pass * S_par);
        const int n_rows = slice < S && g < n_b ? (n_b - g + G - 1) / G : 0;  // of this warp
        if (pass > 0) __syncthreads();  // the previous pass's sums have been read
        const long long seg_off = (long long)slice * a.seg_bytes;
        const int seg_len = max(0, min(a.seg_bytes, row_bytes - int(seg_off)));
        const unsigned char* src = a.packed + ((long long)blockIdx.x + (long long)gridDim.x * g) * a.stride + seg_off;
        int off = int(reinterpret_cast<uintptr_t>(src) & 15);  // of the current row from the 16-byte boundary below it
        f32x2 xr[NVEC][16];
        // the ring of a warp: D staged rows of its slice, one commit group per R rows (empty past the end)
        int issued = 0;
        auto issue = [&]() {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (issued < n_rows) {
                    unsigned char* dst = stage + (issued % D) * a.stage_bytes + (lane << 4);
                    const int mis = int(reinterpret_cast<uintptr_t>(src) & 15);
                    const unsigned char* from = src - mis + (lane << 4);
                    const int left = mis + seg_len - (lane << 4);  // at most 49 pieces: two per lane
                    if (left > 0) cp_async_upto16(dst, from, min(16, left));
                    if (left > 512) cp_async_upto16(dst + 512, from + 512, min(16, left - 512));
                    src += src_step;
                }
                ++issued;
            }
            cp_async_commit();
        };
        auto fill = [&]() {
            for (int i = 0; i < D / R - 1; ++i) issue();
        };
        if (NVEC == 4) fill();  // the ring is free of the rotation: the first rows travel meanwhile
        if (n_rows > 0) {
            if constexpr (NVEC == 4) {
                const bool valid = 32 * slice + lane < a.n_chunks;
#pragma unroll
                for (int v = 0; v < NVEC; ++v)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 q = valid ? __ldcg(a.xt + xt_index(a, slice, v, j, lane)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        xr[v][2 * j] = pack2(q.x, q.y);
                        xr[v][2 * j + 1] = pack2(q.z, q.w);
                    }
            } else {
                // the first rows come to the L2 while the ring's memory serves the rotation
                for (int i = 0; i < min(n_rows, D) && lane * 128 < seg_len + 15; ++i)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(src + i * src_step + min(lane * 128, seg_len - 1)));
                rotate_slice<NVEC>(a, slice, 0, stage, lane, xr);
            }
        }
        if (NVEC != 4) fill();

        for (int tile = 0; tile < n_tiles; ++tile) {
            float* ps = ps_base + (tile & 1) * (S_par * TI * NVEC);  // [slice][row of the tile][vector]
            for (int jj = 0; jj < JT; jj += R) {
                const int it = tile * JT + jj;  // this warp's row counter
                if (it >= n_rows) break;
                cp_async_wait_pending<D / R - 2>();
                __syncwarp();  // every lane's part of these rows has landed; the buffers refilled next are no longer read
                issue();
                // R rows at once; past the last row of the warp the sums of stale bytes are computed and not stored
                uint32_t win[R][NB + 1];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t in = stage_addr + uint32_t(((it + r) % D) * a.stage_bytes) + w_off + uint32_t(off);
                    off = (off + int(src_step & 15)) & 15;
                    uint32_t word[NW + 1];
#pragma unroll
                    for (int i = 0; i < NW; ++i) word[i] = lds_word(in + 4u * i);
                    word[NW] = 0u;
#pragma unroll
                    for (int i = 0; i < NB; ++i) win[r][i] = ODD ? __funnelshift_r(word[i], word[i + 1], sh) : word[i];
                    win[r][NB] = 0u;
                }
                f32x2 acc[R][NVEC];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int v = 0; v < NVEC; ++v) acc[r][v] = 0ull;
#pragma unroll
                for (int t = 0; t < 16; ++t) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        uint32_t id;
                        if (BT) {
                            constexpr int W = BT ? BT : 1;
                            const int w = t * W / 32, s = t * W % 32;
                            id = (s + W <= 32 ? win[r][w] >> s : __funnelshift_r(win[r][w], win[r][w + 1 <= NB ? w + 1 : NB], s)) & mask;
                        } else {
                            const unsigned bit = unsigned(t * B);
                            const uint32_t lo = bit < 32u ? win[r][0] : bit < 64u ? win[r][1] : win[r][2];
                            const uint32_t hi = bit < 32u ? win[r][1] : bit < 64u ? win[r][2] : win[r][3 <= NB ? 3 : NB];
                            id = __funnelshift_r(lo, hi, bit & 31u) & mask;
                        }
                        const float2 c = lds_f32x2(cb + id * cb_stride);
                        const f32x2 c2 = pack2(c.x, c.y);
#pragma unroll
                        for (int v = 0; v < NVEC; ++v) acc[r][v] = fma2(c2, xr[v][t], acc[r][v]);
                    }
                }
                float sums[R * NVEC];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int v = 0; v < NVEC; ++v) {
                        float p, q;
                        unpack2(acc[r][v], p, q);
                        sums[r * NVEC + v] = p + q;
                    }
                const float total = warp_sums<R * NVEC>(sums, lane);
                constexpr int W = 32 / (R * NVEC);
                if (lane % W == 0) {
                    const int id = lane / W, r = id / NVEC, v = id - r * NVEC;
                    if (it + r < n_rows) ps[(s0 * TI + (jj + r) * G + g) * NVEC + v] = total;
                }
            }
            // the norm of this thread's first row travels while the block's warps meet
            const int i0 = tile * TI + int(threadIdx.x) / NVEC;
            float rn = i0 < n_b ? a.row_norm[(long long)blockIdx.x + (long long)gridDim.x * i0] : 0.f;
            __syncthreads();  // the tile's partial sums are complete
            for (int idx = threadIdx.x; idx < TI * NVEC; idx += blockDim.x) {
                const int il = idx / NVEC, v = idx - il * NVEC;
                const int i = tile * TI + il;
                if (i >= n_b) continue;
                const long long row = (long long)blockIdx.x + (long long)gridDim.x * i;
                if (idx >= int(blockDim.x)) rn = a.row_norm[row];
                float sum = 0.f;
                for (int sl = 0; sl < n_live; ++sl) sum += ps[(sl * TI + il) * NVEC + v];
                sum *= rn;
                if (pass == 0) a.y[row * NVEC + v] = sum;
                else a.y[row * NVEC + v] += sum;
            }
        }
        cp_async_wait_all();
    }
}

// The arguments are read where they lie, in constant memory (__grid_constant__), instead of being copied to registers first: at four
// vectors, whose activations take 128 registers, that is 1 to 7 % faster (eleven shapes at K = 64, 256, 2048 and 4096;
// 13824 x 5120, K = 2048: 39.8 -> 38.9 us).  At two vectors the copy stays: without it blocks of few rows take longer (2048 x 5632: 12.0 ->
// 12.5 us), if blocks of many take less (13824 x 5120: 34.2 -> 33.3).
template <int NVEC, int BT>
__global__ void __launch_bounds__(GemvGeom<NVEC>::kThreads, 1) gemv2_kernel(const __grid_constant__ Gemv2Args a) {
    gemv2_rows<NVEC, BT>(a);
}
template <int BT>
__global__ void __launch_bounds__(GemvGeom<2>::kThreads, 1) gemv2_two_kernel(const Gemv2Args a) {
    gemv2_rows<2, BT>(a);
}

int gemv_check(const char* what, cudaError_t e) {
    if (e != cudaSuccess) {
        set_cuda_error(what, int(e));
        return QAMW_ERR_CUDA;
    }
    return QAMW_OK;
}

template <int NVEC>
int launch_gemv(const GemvArgs& a, int blocks, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(gemv_kernel<NVEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemLimit));
    if (e != cudaSuccess) {
        set_cuda_error("cudaFuncSetAttribute", int(e));
        return QAMW_ERR_NOMEM;
    }
    return gemv_check("gemv_kernel", launch_chained(gemv_kernel<NVEC>, blocks, 512, smem, st, a));
}

// cudaFuncSetAttribute once per kernel and device
int gemv_raise_smem(const void* kernel) {
    static std::mutex mu;
    static std::unordered_map<const void*, unsigned long long> done;
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    std::lock_guard<std::mutex> lock(mu);
    unsigned long long& m = done[kernel];
    if (m & bit) return QAMW_OK;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemLimit));
    if (e != cudaSuccess) {
        set_cuda_error("cudaFuncSetAttribute", int(e));
        return QAMW_ERR_NOMEM;
    }
    m |= bit;
    return QAMW_OK;
}

template <int NVEC, int BT>
int launch_gemv2_b(const Gemv2Args& a, int blocks, int threads, size_t smem, cudaStream_t st) {
    auto go = [&](auto* kernel) {
        int rc = gemv_raise_smem(reinterpret_cast<const void*>(kernel));
        return rc ? rc : gemv_check("gemv2_kernel", launch_chained(kernel, blocks, threads, smem, st, a));
    };
    if constexpr (NVEC == 2) return go(&gemv2_two_kernel<BT>);
    else return go(&gemv2_kernel<NVEC, BT>);
}

template <int NVEC>
int launch_gemv2(const Gemv2Args& a, int sms, cudaStream_t st) {
    constexpr int kThreads = GemvGeom<NVEC>::kThreads, kWarps = kThreads / 32;
    // as many passes as the warps of a block require, the slices spread evenly over them
    const int passes = (a.n_slices + kWarps - 1) / kWarps;
    const int S_par = (a.n_slices + passes - 1) / passes;
    const int blocks = std::max(1, std::min(sms, a.d_out));
    const int n_b = (a.d_out + blocks - 1) / blocks;  // rows of a block
    const int G = std::max(1, std::min(kWarps / S_par, n_b));
    Gemv2Args b = a;
    b.s_par = S_par;
    b.log2c = pick_copies(a.K, (long long)n_b * (a.d_in / 64), size_t(128) * 1024);
    const int threads = 32 * S_par * G;
    const size_t sums = size_t(2) * S_par * GemvGeom<NVEC>::kTileRows * G * NVEC * sizeof(float);
    const size_t smem = (size_t(a.K) * 8 << b.log2c) + size_t(S_par * G) * GemvGeom<NVEC>::kDepth * a.stage_bytes + sums;
    if (smem > kSmemLimit) return QAMW_ERR_NOMEM;
    switch (a.B) {
        case 6: return launch_gemv2_b<NVEC, 6>(b, blocks, threads, smem, st);
        case 7: return launch_gemv2_b<NVEC, 7>(b, blocks, threads, smem, st);
        case 8: return launch_gemv2_b<NVEC, 8>(b, blocks, threads, smem, st);
        case 9: return launch_gemv2_b<NVEC, 9>(b, blocks, threads, smem, st);
        case 10: return launch_gemv2_b<NVEC, 10>(b, blocks, threads, smem, st);
        case 11: return launch_gemv2_b<NVEC, 11>(b, blocks, threads, smem, st);
        case 12: return launch_gemv2_b<NVEC, 12>(b, blocks, threads, smem, st);
        default: return launch_gemv2_b<NVEC, 0>(b, blocks, threads, smem, st);
    }
}

int gemv_slices(int d_in) { return (d_in / 32 + 31) / 32; }

}  // namespace

extern "C" size_t qamw_gemv_workspace_bytes(const qamw_params* p, int n_vec) {
    if (check_matrix_params(p) || n_vec < 1) return 0;
    return size_t(n_vec) * size_t(p->d_in) * sizeof(float);  // rotated activations
}

extern "C" int qamw_decode_gemv(const uint8_t* packed, const float* row_norm, const float* chan_scale,
                                const int8_t* signs, const float* sigma, const qamw_codebook* cb, const qamw_params* p,
                                const float* x, int n_vec, float* y_out, void* workspace, size_t workspace_bytes,
                                void* stream) {
    int rc = check_matrix_params(p);
    if (rc) return rc;
    if (!packed || !row_norm || !signs || !sigma || !cb || !x || !y_out || !workspace) return QAMW_ERR_ARG;
    if (cb->K != p->K) return QAMW_ERR_ARG;
    if (n_vec != 1 && n_vec != 2 && n_vec != 4) return QAMW_ERR_ARG;
    if (p->d_in % 32) return QAMW_ERR_SHAPE;  // whole chunks of 16 pairs
    const size_t row_bytes = qamw_packed_row_bytes(p->d_in, p->K);
    if (p->packed_row_stride < (long long)row_bytes || p->packed_row_stride % 4) return QAMW_ERR_ALIGN;
    if (reinterpret_cast<uintptr_t>(packed) % 4 || reinterpret_cast<uintptr_t>(workspace) % 8) return QAMW_ERR_ALIGN;
    if (workspace_bytes < qamw_gemv_workspace_bytes(p, n_vec)) return QAMW_ERR_NOMEM;
    if (p->d_out == 0) return QAMW_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool general = (p->flags & QAMW_FLAG_GENERAL_KERNELS) != 0;
    auto aligned16 = [](const void* v) { return reinterpret_cast<uintptr_t>(v) % 16 == 0; };
    if (!general && aligned16(packed) && aligned16(workspace) && aligned16(x) && aligned16(chan_scale) && aligned16(signs) && aligned16(sigma)) {
        Gemv2Args g{};
        g.packed = packed;
        g.stride = p->packed_row_stride;
        g.x = x;
        g.chan_scale = chan_scale;
        g.signs = signs;
        g.sigma = sigma;
        g.codebook = static_cast<const float2*>(cb->d_blob);
        g.row_norm = row_norm;
        g.y = y_out;
        g.d_out = p->d_out;
        g.d_in = p->d_in;
        g.n_chunks = p->d_in / 32;
        g.n_slices = gemv_slices(p->d_in);
        g.K = p->K;
        g.B = ilog2(p->K);
        g.log2b = ilog2(p->block);
        g.seg_bytes = 64 * g.B;
        // 12 bytes before a row off its boundary, 4 read past the last lane's indices; the ring also serves rotate_slice
        g.stage_bytes = std::max((g.seg_bytes + 32 + 127) & ~127, kRotateStage / GemvGeom<1>::kDepth);
        g.xt = static_cast<float4*>(workspace);
        g.inv_sqrt_b = 1.0f / std::sqrt(float(p->block));
        const int sms = sm_count();
        if (n_vec == 1) return launch_gemv2<1>(g, sms, st);
        if (n_vec == 2) return launch_gemv2<2>(g, sms, st);
        // Four vectors are rotated once by a small kernel of its own: done by every block, as for one or two, it
        // costs 650 wavefronts per warp and the registers that the rows need.
        rc = gemv_check("gemv_rotate4_kernel", launch_chained(gemv_rotate4_kernel, g.n_slices, 32 * kRotateWarps, 0, st, g));
        return rc ? rc : launch_gemv2<4>(g, sms, st);
    }
    const size_t x_bytes = size_t(n_vec) * p->d_in * sizeof(float);
    if (x_bytes + size_t(p->K) * 8 > kSmemLimit || size_t(p->d_in) * sizeof(float) > kSmemLimit) return QAMW_ERR_NOMEM;
    float2* xt = static_cast<float2*>(workspace);
    if (size_t(p->d_in) * sizeof(float) > 48 * 1024) {  // beyond the default dynamic limit
        cudaError_t e = cudaFuncSetAttribute(gemv_rotate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemLimit));
        if (e != cudaSuccess) {
            set_cuda_error("cudaFuncSetAttribute", int(e));
            return QAMW_ERR_NOMEM;
        }
    }
    rc = gemv_check("gemv_rotate_kernel", launch_chained(gemv_rotate_kernel, n_vec, 1024, size_t(p->d_in) * sizeof(float), st, x,
                                                         chan_scale, signs, sigma, p->d_in, ilog2(p->block), xt));
    if (rc) return rc;
    GemvArgs a;
    a.packed = packed;
    a.stride = p->packed_row_stride;
    a.row_norm = row_norm;
    a.codebook = static_cast<const float2*>(cb->d_blob);
    a.xt = xt;
    a.y = y_out;
    a.d_out = p->d_out;
    a.n_pairs = p->d_in / 2;
    a.K = p->K;
    a.B = ilog2(p->K);
    a.log2c = 4;
    while (a.log2c > 0 && (size_t(p->K) * 8 << a.log2c) + x_bytes > std::min(kSmemLimit, size_t(128) * 1024 + x_bytes)) --a.log2c;
    const size_t smem = (size_t(p->K) * 8 << a.log2c) + x_bytes;
    const int blocks = std::max(1, std::min(sm_count(), (p->d_out + 15) / 16));
    if (n_vec == 1) return launch_gemv<1>(a, blocks, smem, st);
    if (n_vec == 2) return launch_gemv<2>(a, blocks, smem, st);
    return launch_gemv<4>(a, blocks, smem, st);
}
