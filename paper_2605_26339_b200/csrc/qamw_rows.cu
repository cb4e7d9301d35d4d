// Row kernels of libqamw for the common layouts (16-byte aligned rows of W, d_in a multiple of 8): one persistent launch
// walks any number of matrices.
//
// Geometry.
//   * A warp owns a "segment" of 256 * NS consecutive elements of a row: NS = 4 octets (32 elements)
//     per thread in the decoder, NS = 2 (16 elements) in the encoder, whose register budget then
//     allows up to 28 resident warps per SM (16 to 28 by row length, see encode_warps).  A row is owned by a group of
//     ceil(d_in / (256 NS)) warps; a block holds as many groups as fit and the grid is persistent.
//   * A launch takes an array of matrix descriptors.  The rows of all matrices form one list, cut
//     into one contiguous span per block with (nearly) equal numbers of weights, so a block meets one
//     or two matrices; the tables in shared memory (codebook copies, cell records) are filled once
//     per launch and only the per-column constants of a warp's segment are reloaded when the matrix
//     changes.
//   * Walsh-Hadamard butterflies of a block of b elements: stages h = 1, 2, 4 inside an octet, then
//     one stage per octet slot bit inside the thread, then one "half exchange" per lane bit: a thread
//     keeps the slots whose top slot bit is 0, sends the others to its partner (lane ^ 2^j), and
//     computes both outputs (K + R, K - R) of the butterflies whose inputs it then holds.  Every
//     exchange uses the top slot bit, so after the last stage a thread holds runs of NS/2 adjacent
//     octets and the threads of a block cover consecutive runs: 32-byte stores that tile full
//     128-byte lines (decoder).  A thread starts with NS consecutive octets.  Which physical slot
//     receives the sum and which the difference of a stage is chosen so that the next stage can again
//     keep the lower slots and send the upper ones without moving registers: a thread whose next lane
//     bit is set multiplies the received value by -1 first (K - R, K + R), and the last in-thread
//     stage does the same for odd lanes.  An upper partner then holds R - K as K - R: some slots end
//     up negated, by a pattern that depends on the lane only and is folded into the per-column
//     constants.  Stages run in ascending order of h with one f32 rounding per output, and a
//     multiplication by +-1 is exact, so the result is bit-identical to the plain butterfly.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "qamw_device.cuh"
#include "qamw_internal.h"
#include "qamw_launch.h"

using namespace qamw;

namespace {

// ---------------------------------------------------------------------------------------------
// layout of a Hadamard block over NS slots and L = 2^S lanes
// ---------------------------------------------------------------------------------------------
// LOG2B = 0: blocks of 2 to 16 elements, whose size is a run-time value; they never leave the thread.
template <int NS, int LOG2B>
struct Lay2 {
    static_assert(NS == 2 || NS == 4, "two or four octets per thread");
    static constexpr int LS = NS == 4 ? 2 : 1;          // slot bits
    static constexpr int TOP = NS / 2;                  // value of the top slot bit
    static constexpr int S = LOG2B ? LOG2B - 3 - LS : 0;  // cross-lane stages
    static_assert(S >= 0 && S <= 5, "block size out of range for this geometry");
    static constexpr int L = 1 << S;
    // octet (units of 8 elements, relative to the warp's segment) in physical slot p before the
    // butterflies: NS consecutive octets per lane
    __device__ static __forceinline__ int octet_before(int lane, int p) { return NS * lane + p; }
    // ... and after them
    __device__ static __forceinline__ int octet_after(int lane, int p) {
        if (S == 0) return NS * lane + p;
        const int q = lane & (L - 1), blk = lane >> S;
        const int o = (p & (TOP - 1)) | ((q & 1) << (LS - 1)) | ((q >> 1) << LS) | ((p >> (LS - 1)) << (LS + S - 1));
        return blk * (NS * L) + o;
    }
    // true if physical slot p of this lane holds minus the butterfly output
    __device__ static __forceinline__ bool negated(int lane, int p) {
        bool neg_k = false, neg_x = false;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const bool upper = (lane >> j) & 1;
            const bool normal = (j == S - 1) || !((lane >> (j + 1)) & 1);
            if (normal) {
                neg_x = neg_k ^ upper;
            } else {
                const bool old = neg_k;
                neg_k = old ^ upper;
                neg_x = old;
            }
        }
        return (p & TOP) ? neg_x : neg_k;
    }
};

// Unnormalised Walsh-Hadamard butterfly of the NS x 8 elements of a thread and, for wider blocks, of
// the L lanes of the block.  P[p][i] holds elements (2i, 2i+1) of the octet in physical slot p.
// FIRST_STAGE_DONE: the caller's inputs already went through stage h = 1.
template <int NS, int LOG2B, bool FIRST_STAGE_DONE>
__device__ __forceinline__ void fwht2(f32x2 (&P)[NS][4], int lane, int log2b_small) {
    typedef Lay2<NS, LOG2B> Lay;
    constexpr int TOP = Lay::TOP;
    if (!FIRST_STAGE_DONE) {
#pragma unroll
        for (int p = 0; p < NS; ++p)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float a, c;
                unpack2(P[p][i], a, c);
                P[p][i] = pack2(__fadd_rn(a, c), __fsub_rn(a, c));
            }
    }
    if constexpr (LOG2B == 0) {
#pragma unroll
        for (int p = 0; p < NS; ++p) {
            if (log2b_small >= 2) {
                bfly2(P[p][0], P[p][1]);
                bfly2(P[p][2], P[p][3]);
            }
            if (log2b_small >= 3) {
                bfly2(P[p][0], P[p][2]);
                bfly2(P[p][1], P[p][3]);
            }
        }
        if (log2b_small >= 4) {
#pragma unroll
            for (int p = 0; p < NS; p += 2)
#pragma unroll
                for (int i = 0; i < 4; ++i) bfly2(P[p][i], P[p + 1][i]);
        }
    } else {
#pragma unroll
    for (int p = 0; p < NS; ++p) {  // h = 2, 4
        bfly2(P[p][0], P[p][1]);
        bfly2(P[p][2], P[p][3]);
        bfly2(P[p][0], P[p][2]);
        bfly2(P[p][1], P[p][3]);
    }
    if (NS == 4) {  // h = 8: slot bit 0
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            bfly2(P[0][i], P[1][i]);
            bfly2(P[2 % NS][i], P[3 % NS][i]);
        }
    }
    // top slot bit (h = 8 for NS = 2, h = 16 for NS = 4).  The first half exchange wants the two
    // halves of an odd lane in swapped places, so an odd lane writes its difference into the lower
    // slots and its sum into the upper ones: out_lo = a + s c, out_hi = a - s c with s = -1.
    if (Lay::S >= 1) {
        const float s0 = (lane & 1) ? -1.0f : 1.0f;
        const f32x2 sp = pack2(s0, s0), sn = pack2(-s0, -s0);
#pragma unroll
        for (int p = 0; p < TOP; ++p)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const f32x2 a = P[p][i], c = P[p + TOP][i];
                P[p][i] = fma2(c, sp, a);
                P[p + TOP][i] = fma2(c, sn, a);
            }
    } else {
#pragma unroll
        for (int p = 0; p < TOP; ++p)
#pragma unroll
            for (int i = 0; i < 4; ++i) bfly2(P[p][i], P[p + TOP][i]);
    }
    // cross-lane stages
#pragma unroll
    for (int j = 0; j < Lay::S; ++j) {
        if (j == Lay::S - 1) {
#pragma unroll
            for (int p = 0; p < TOP; ++p)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f32x2 keep = P[p][i];
                    const f32x2 got = shfl_xor2(P[p + TOP][i], 1 << j);
                    P[p][i] = add2(keep, got);
                    P[p + TOP][i] = sub2(keep, got);
                }
        } else {
            const float al = ((lane >> (j + 1)) & 1) ? -1.0f : 1.0f;
            const f32x2 ap = pack2(al, al), an = pack2(-al, -al);
#pragma unroll
            for (int p = 0; p < TOP; ++p)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f32x2 keep = P[p][i];
                    const f32x2 got = shfl_xor2(P[p + TOP][i], 1 << j);
                    P[p][i] = fma2(got, ap, keep);
                    P[p + TOP][i] = fma2(got, an, keep);
                }
        }
    }
    }  // LOG2B != 0
}

__device__ __forceinline__ void st_global_256(void* p, const uint32_t (&w)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                 "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
__device__ __forceinline__ void ld_global_256(const void* p, uint32_t (&w)[8]) {
    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(p));
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// The span of the concatenated row list that this block works on: first matrix, first row in it,
// last matrix, end row in it.  Without a span table there is one matrix, split evenly.
__device__ __forceinline__ int4 block_span(const int4* spans, int d_out_single) {
    if (spans) return spans[blockIdx.x];
    const long long n = d_out_single;
    return make_int4(0, int(n * blockIdx.x / gridDim.x), 0, int(n * (blockIdx.x + 1) / gridDim.x));
}

// Per-column constants of a thread's octets, as they lie in memory: scales and signs of octet e[p], pair scales of octet
// k[p].  All loads are issued before the first is used, and none depends on a test (an octet lies inside the row or outside: d_in
// is a multiple of 8; one outside reads the first and is masked by its user): loads behind tests of their own came one after the
// other, 1.0 us for two octets and 4.4 us for four, before the first row was asked for.
template <int NS, bool SIGMA>
struct Columns {
    float4 cs[NS][2], sg[SIGMA ? NS : 1];
    uint2 sign[NS];
    __device__ __forceinline__ void load(const float* chan_scale, const int8_t* signs, const float* sigma, const int (&e)[NS], const int (&k)[NS],
                                         int d_in) {
#pragma unroll
        for (int p = 0; p < NS; ++p) {
            sign[p] = *reinterpret_cast<const uint2*>(signs + (8 * e[p] < d_in ? 8 * e[p] : 0));
            if (SIGMA) sg[SIGMA ? p : 0] = *reinterpret_cast<const float4*>(sigma + (8 * k[p] < d_in ? 4 * k[p] : 0));
        }
        if (chan_scale) {
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                const float4* c = reinterpret_cast<const float4*>(chan_scale + (8 * e[p] < d_in ? 8 * e[p] : 0));
                cs[p][0] = c[0];
                cs[p][1] = c[1];
            }
        } else {
#pragma unroll
            for (int p = 0; p < NS; ++p) cs[p][0] = cs[p][1] = make_float4(1.f, 1.f, 1.f, 1.f);
        }
    }
    // scales (1 outside the row) and signs (0 outside)
    __device__ __forceinline__ void unpack(int p, bool in, float (&c)[8], float (&s)[8]) const {
        const float4 a = cs[p][0], b = cs[p][1];
        const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t byte = ((i < 4 ? sign[p].x : sign[p].y) >> (8 * (i & 3))) & 0xffu;
            c[i] = in ? v[i] : 1.0f;
            s[i] = in ? __uint_as_float(0x3f800000u | ((byte & 0x80u) << 24)) : 0.f;  // +-1.0f from the byte's sign bit
        }
    }
};

// ---------------------------------------------------------------------------------------------
// decoder
// ---------------------------------------------------------------------------------------------
constexpr int kDecodeDepth = 4;

struct Decode2Args {
    const MatDesc* descs;    // device array, or NULL: `one` is the only matrix
    MatDesc one;
    const int4* spans;       // per block (see block_span), or NULL
    const float2* codebook;  // device, K entries
    int K, log2K, log2c;
    int seg_bytes;           // packed bytes of one warp segment: 16 * NS * B
    int stage_bytes;         // one staging buffer of a warp (128-byte aligned, at least seg_bytes + 28)
    int log2b;               // log2 of the Hadamard block
    float inv_sqrt_b;
};

// A warp streams its segment of the packed row through its own shared-memory ring of kDecodeDepth rows
// (16-byte asynchronous copies, kDecodeDepth - 1 rows ahead: with one row in flight per warp the reads
// are bound by memory latency); nothing is shared between warps after the prologue, so there is no
// barrier.  A row that starts off a 16-byte boundary is copied from the boundary below it and read at an offset.
// Per row a thread reads its 4 NS B index bits as two runs of 32-bit words, gathers the codewords
// (stored as (x + y, x - y): butterfly stage h = 1) from its own bank-separated copy, scales them by
// the pair scales, runs the remaining butterflies and writes bf16.
// ALIGNED: packed rows start on 16 bytes, rows of the output on 32, d_in is a multiple of 16.
constexpr int kDecodeSlots = 4, kDecodeWarps = 16;  // octets per thread; warps of a block at most
template <int LOG2B, bool ALIGNED>
__global__ void __launch_bounds__(32 * kDecodeWarps, 1) decode2_kernel(const Decode2Args a) {
    constexpr int NS = kDecodeSlots;
    typedef Lay2<NS, LOG2B> Lay;
    constexpr int TOP = Lay::TOP;
    constexpr int WE = 256 * NS;  // elements of a warp segment
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int B = a.log2K;
    const uint32_t mask = (1u << B) - 1u;
    const uint32_t cb_stride = 8u << a.log2c;
    const uint32_t cb = smem_addr(smem) + 8u * (threadIdx.x & ((1 << a.log2c) - 1));
    unsigned char* stage = smem + ((size_t(a.K) * 8) << a.log2c) + size_t(warp) * kDecodeDepth * a.stage_bytes;
    const uint32_t stage_addr = smem_addr(stage);

    chain_release();
    fill_codebook_copies(reinterpret_cast<float2*>(smem), a.codebook, a.K, a.log2c, true);
    // spans and descriptors are written once, before the batch handle exists: what follows from them comes before the wait
    const int4 span = block_span(a.spans, a.one.d_out);
    __syncthreads();

    // where this thread's index bits sit inside a staged segment: two runs (the lower and the upper
    // physical slots), each 4 B TOP bits long
    uint32_t run_word[2], run_shift[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const unsigned bit0 = unsigned(4 * Lay::octet_before(lane, x * TOP)) * unsigned(B);
        run_word[x] = 4u * (bit0 >> 5);
        run_shift[x] = bit0 & 31u;
    }

    bool waited = false;
    for (int m = span.x; m <= span.z; ++m) {
        const MatDesc& d = a.descs ? a.descs[m] : a.one;
        const int d_in = d.d_in, n_pairs = d_in >> 1;
        const int row_begin = m == span.x ? span.y : 0;
        const int row_end = m == span.z ? span.w : d.d_out;
        const int n_seg = (d_in + WE - 1) / WE;
        const int groups = n_warps / n_seg;  // >= 1 (checked on the host)
        const int group = warp / n_seg, seg = warp - group * n_seg;
        const int row0 = row_begin + group;
        if (group >= groups || row0 >= row_end) continue;  // this warp has no work in this matrix
        const int row_step = groups;
        const int n_rows = (row_end - row0 + row_step - 1) / row_step;
        const long long pstride = d.packed_row_stride;
        constexpr int kGran = ALIGNED ? 16 : 4;  // of row starts: the stride is a multiple of it, and a row may be read up to one
        const int row_bytes = int((((long long)n_pairs * B + 7) / 8 + kGran - 1) & ~(long long)(kGran - 1));
        const long long seg_off = (long long)seg * a.seg_bytes;
        const int seg_len = max(0, min(a.seg_bytes, row_bytes - int(seg_off)));
        const unsigned char* src = d.packed + (long long)row0 * pstride + seg_off;  // next row to fetch
        const long long src_step = (long long)row_step * pstride;
        uint32_t off = ALIGNED ? 0u : uint32_t(reinterpret_cast<uintptr_t>(src) & 15);  // of the row decoded next from the boundary below it
        const uint32_t off_step = ALIGNED ? 0u : uint32_t(src_step & 15);
        const bool copy0 = (lane << 4) < seg_len, copy1 = (lane << 4) + 512 < seg_len;  // two pieces of 16 bytes per lane, no loop
        if (!waited) chain_wait();
        waited = true;
        int issued = 0;
        auto issue_row = [&]() {  // one commit group per row, empty past the end
            if (issued < n_rows) {
                unsigned char* dst = stage + (issued % kDecodeDepth) * a.stage_bytes + (lane << 4);
                if constexpr (ALIGNED) {
                    if (copy0) cp_async(dst, src + (lane << 4), 4);
                    if (copy1) cp_async(dst + 512, src + (lane << 4) + 512, 4);
                } else {
                    const int mis = int(reinterpret_cast<uintptr_t>(src) & 15);
                    const unsigned char* from = src - mis + (lane << 4);
                    const int left = mis + seg_len - (lane << 4);
                    if (left > 0) cp_async_upto16(dst, from, min(16, left));
                    if (left > 512) cp_async_upto16(dst + 512, from + 512, min(16, left - 512));
                }
                src += src_step;
            }
            ++issued;
            cp_async_commit();
        };
        __syncwarp();  // the previous matrix's last row has been read by every lane
        for (int i = 0; i < kDecodeDepth - 1; ++i) issue_row();

        // per-column constants of this warp's segment
        const int oct0 = seg * (WE / 8);  // first octet of the segment
        float sg[NS][4];
        f32x2 mcol[NS][4];
        int e_out[NS], e_oct[NS], k_oct[NS];
#pragma unroll
        for (int p = 0; p < NS; ++p) {
            k_oct[p] = oct0 + Lay::octet_before(lane, p);
            e_oct[p] = oct0 + Lay::octet_after(lane, p);
        }
        Columns<NS, true> cols;
        cols.load(d.chan_scale, d.signs, d.sigma, e_oct, k_oct, d_in);
        const f32x2 c2 = pack2(a.inv_sqrt_b, a.inv_sqrt_b);
#pragma unroll
        for (int p = 0; p < NS; ++p) {
            const bool in = 8 * k_oct[p] < d_in;  // a pair beyond the row has scale 0
            const float4 v = cols.sg[p];
            sg[p][0] = in ? v.x : 0.f;
            sg[p][1] = in ? v.y : 0.f;
            sg[p][2] = in ? v.z : 0.f;
            sg[p][3] = in ? v.w : 0.f;
            e_out[p] = 8 * e_oct[p];
            float cs[8], sgn[8];
            cols.unpack(p, e_out[p] < d_in, cs, sgn);
            const float fl = Lay::negated(lane, p) ? -1.0f : 1.0f;
            uint32_t off = 0;  // a scale that quotient2 does not take
#pragma unroll
            for (int i = 0; i < 8; ++i) off |= uint32_t(__float_as_uint(cs[i]) - 0x21800000u >= 0x3c000000u);  // [2^-60, 2^60)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                f32x2 v = quotient2(c2, cs[2 * i], cs[2 * i + 1]);
                if (off) v = pack2(library_quotient(a.inv_sqrt_b, cs[2 * i]), library_quotient(a.inv_sqrt_b, cs[2 * i + 1]));
                mcol[p][i] = mul2(pack2(fl * sgn[2 * i], fl * sgn[2 * i + 1]), v);
            }
        }
        __nv_bfloat16* orow = static_cast<__nv_bfloat16*>(d.w_hat) + (long long)row0 * d_in;
        const long long out_step = (long long)row_step * d_in;
        const float* rnp = d.row_norm + row0;

        for (int it = 0; it < n_rows; ++it, orow += out_step, rnp += row_step) {
            const float rn = *rnp;
            cp_async_wait_pending<kDecodeDepth - 2>();
            __syncwarp();  // every lane's part of this row has landed; the buffer refilled next is no longer read
            issue_row();
            const uint32_t in = stage_addr + uint32_t((it % kDecodeDepth) * a.stage_bytes) + off;
            if (!ALIGNED) off = (off + off_step) & 15u;
            f32x2 P[NS][4];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const uint32_t w = in + run_word[x];
                const uint32_t sh = run_shift[x];
                uint32_t id[4 * TOP];
                // 8 indices = 8 B bits <= 96: four words, shifted down to three, then cut in steps of 2 B bits
                const uint32_t w0 = lds_u32(w), w1 = lds_u32(w + 4), w2 = lds_u32(w + 8), w3 = lds_u32(w + 12);
                uint32_t v0 = __funnelshift_r(w0, w1, sh), v1 = __funnelshift_r(w1, w2, sh), v2 = __funnelshift_r(w2, w3, sh);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    id[2 * t] = v0 & mask;
                    id[2 * t + 1] = (v0 >> B) & mask;
                    if (t < 3) {
                        v0 = __funnelshift_r(v0, v1, 2 * B);
                        v1 = __funnelshift_r(v1, v2, 2 * B);
                        v2 >>= 2 * B;
                    }
                }
#pragma unroll
                for (int t = 0; t < TOP; ++t) {
                    const int p = x * TOP + t;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // pairs beyond the end of the row have scale 0 and decode to 0 whatever their bits are
                        const float2 c = lds_f32x2(cb + id[4 * t + i] * cb_stride);
                        P[p][i] = pack2(c.x * sg[p][i], c.y * sg[p][i]);
                    }
                }
            }
            fwht2<NS, LOG2B, true>(P, lane, a.log2b);
            const f32x2 rn2 = pack2(rn, rn);
#pragma unroll
            for (int p = 0; p < NS; p += 2) {
                constexpr int NP = 2;  // adjacent octets written by one store
                uint32_t w[4 * NP];
#pragma unroll
                for (int t = 0; t < NP; ++t)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float y0, y1;
                        unpack2(mul2(P[p + t][i], mul2(mcol[p + t][i], rn2)), y0, y1);
                        __nv_bfloat162 h2 = __floats2bfloat162_rn(y0, y1);
                        w[4 * t + i] = *reinterpret_cast<uint32_t*>(&h2);
                    }
                if constexpr (ALIGNED) {
                    if (e_out[p] < d_in) st_global_256(orow + e_out[p], w);
                } else {
#pragma unroll
                    for (int t = 0; t < NP; ++t)
                        if (e_out[p + t] < d_in)
                            *reinterpret_cast<uint4*>(orow + e_out[p + t]) = make_uint4(w[4 * t], w[4 * t + 1], w[4 * t + 2], w[4 * t + 3]);
                }
            }
        }
        cp_async_wait_all();
    }
}

// ---------------------------------------------------------------------------------------------
// encoder
// ---------------------------------------------------------------------------------------------
struct Encode2Args {
    const MatDesc* descs;
    MatDesc one;
    const int4* spans;
    const float2* codebook;  // device, K entries
    const uint4* table;      // cells | overflow, as laid out by qamw_codebook_create
    int table_bytes;         // a multiple of 16
    int off_overflow;        // byte offset inside the table
    int K, log2K, grid;
    f32x2 map_zlo, map_c0, map_c1, map_c2, map_bias;  // the cell map of the table, each value twice
    int log2c;               // log2 of the number of codebook copies in shared memory
    int log2b;               // log2 of the Hadamard block
    int wide;                // rows of W start on 32 bytes and d_in is a multiple of 8 NS
    int brute;               // every point is compared with the whole codebook
    float reach;             // |z| from which on a point is: 16000, or -1 with `brute`
    float inv_sqrt_b;        // c_b = f32(1 / sqrt(b))
    int32_t* status;         // out (optional): bit 0 set when a row norm is not finite
    unsigned char* calib_base;  // calibration mode: base of the partial-sum workspace (MatDesc::calib_offset)
    int polar_ba, polar_bp;  // polar quantiser: amplitude and phase bits; `table` then holds the squared
                             // amplitude thresholds (2^Ba floats) and, from off_overflow on, the unit vectors
                             // of the phase bin boundaries of the upper half plane (2^Bp / 2 float2)
};

// Polar quantiser (Section 3.5): amplitude |z| to the nearest of 2^Ba levels, phase to one of 2^Bp
// uniform bins, index = (phase << Ba) | amplitude.  Both are binary searches over small tables in
// shared memory: squared thresholds (midpoints of adjacent levels) for the amplitude, and for the
// phase the sign of the cross product with the boundary directions after folding the lower half plane
// onto the upper one.  A point on a threshold takes the lower level, a point on a boundary the bin
// that starts there, the origin bin 0 -- the oracle's rules; within f32 rounding of a threshold or a
// boundary either neighbour may come out.
struct PolarSmem {
    uint32_t thr2;  // shared-memory address of the squared thresholds
    uint32_t bnd;   // ... of the boundary unit vectors
    int Ba, Bp;
};
__device__ __forceinline__ int search_polar(const PolarSmem& s, float zx, float zy) {
    const float r2 = __fmaf_rn(zy, zy, __fmul_rn(zx, zx));
    int a = 0;
    for (int step = (1 << s.Ba) >> 1; step > 0; step >>= 1) {
        float t;
        asm("ld.shared.f32 %0, [%1];" : "=f"(t) : "r"(s.thr2 + 4u * uint32_t(a + step - 1)));
        if (r2 > t) a += step;
    }
    int p = 0;
    if (s.Bp > 0) {
        const bool lower = zy < 0.f || (zy == 0.f && zx < 0.f);
        const float x = lower ? -zx : zx, y = lower ? -zy : zy;
        for (int step = (1 << s.Bp) >> 2; step > 0; step >>= 1) {
            const float2 b = lds_f32x2(s.bnd + 8u * uint32_t(p + step));
            if (__fmaf_rn(b.x, y, -__fmul_rn(b.y, x)) >= 0.f) p += step;
        }
        if (lower) p += (1 << s.Bp) >> 1;
        if (r2 == 0.f) p = 0;
    }
    return (p << s.Ba) | a;
}

// Sum of v over the warp, in every lane, by two 8x8x4 double matrix products with a matrix of ones: the first
// adds the four lanes of a quad, the second the eight quads (two of them added by hand in between).  Ten
// shuffles and five additions, the alternative, load the pipe that binds the encoder.
__device__ __forceinline__ double warp_total(double v) {
    auto quads = [](double b, double& d0, double& d1) {
        asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%4, %4};"
            : "=d"(d0), "=d"(d1)
            : "d"(1.0), "d"(b), "d"(0.0));
    };
    double d0, d1, e0, e1;
    quads(v, d0, d1);          // this lane: totals of quads 2 (lane mod 4) and 2 (lane mod 4) + 1
    quads(d0 + d1, e0, e1);
    return e0;
}

// For every unit of a thread the unit that follows it in the row: units u0 and u1 of a lane lie L units apart, at q
// and q + L of the block (q: lane inside the block).  A lane that is read for its u1 by the last lane of its block is
// not read for its u0, so one shuffle per 32 bits serves both.
template <int L>
__device__ __forceinline__ void next_units(uint32_t u0, uint32_t u1, int lane, uint32_t& n0, uint32_t& n1) {
    const int q = lane & (L - 1);
    const bool first = q == 0, last = q == L - 1;
    n0 = __shfl_sync(kFull, first ? u1 : u0, last ? lane - (L - 1) : lane + 1);
    n1 = __shfl_sync(kFull, first ? u0 : u1, lane + 1);
}

// The words of the packed row that start inside an octet of this thread.  u[p]: the 4 B bits of the octet in
// slot p; first[p]: the first such word (relative to the warp's segment) and, from bit 16 on, its distance from
// the octet's first bit; limit: words of the row's payload from the segment's first on.  The bits past an octet come
// from the lanes that hold the next ones.
template <int NS, int LOG2B>
__device__ __forceinline__ void store_indices(const uint2 (&u)[NS], const uint32_t (&first)[NS], int B, uint32_t* out, int limit, int lane) {
    constexpr int L = Lay2<NS, LOG2B>::L, X = NS / 2;  // the octets that change lanes: slots 0 and X hand over to X - 1 and NS - 1
    const int U = 4 * B;
    if (U > 32) {
        uint2 nxt[NS];
        next_units<L>(u[0].x, u[X].x, lane, nxt[X - 1].x, nxt[NS - 1].x);
        next_units<L>(u[0].y, u[X].y, lane, nxt[X - 1].y, nxt[NS - 1].y);
        if (NS == 4) {
            nxt[0] = u[1 % NS];
            nxt[2 % NS] = u[3 % NS];
        }
#pragma unroll
        for (int p = 0; p < NS; ++p) {
            const int w = int(first[p] & 0xffffu), off = int(first[p] >> 16);
            const uint32_t x1 = u[p].y | (nxt[p].x << (U - 32));
            const uint32_t x2 = __funnelshift_r(nxt[p].x, nxt[p].y, 64 - U);
            if (w < limit) out[w] = __funnelshift_r(u[p].x, x1, off);
            if (off + 32 < U && w + 1 < limit) out[w + 1] = __funnelshift_r(x1, x2, off);
        }
    } else {
        uint32_t cur[NS];
        unsigned long long acc[NS];
#pragma unroll
        for (int p = 0; p < NS; ++p) acc[p] = cur[p] = u[p].x;
        for (int at = U; at < U + 31; at += U) {  // a word that starts in the octet's last bit ends 31 bits later
            uint32_t nxt[NS];
            next_units<L>(cur[0], cur[X], lane, nxt[X - 1], nxt[NS - 1]);
            if (NS == 4) {
                nxt[0] = cur[1 % NS];
                nxt[2 % NS] = cur[3 % NS];
            }
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                cur[p] = nxt[p];
                acc[p] |= (unsigned long long)cur[p] << at;
            }
        }
#pragma unroll
        for (int p = 0; p < NS; ++p) {
            const int w = int(first[p] & 0xffffu), off = int(first[p] >> 16);
            if (off < U && w < limit) out[w] = uint32_t(acc[p] >> off);
        }
    }
}

// Encoder.  A warp owns 256 NS consecutive elements of a row (NS = 2; blocks of 1024 elements take NS = 4): it scales
// them, adds up its part of the row norm, rotates (shuffles only), and after the one meeting point of the
// row's warps -- a named barrier for the norm -- searches its pairs and writes its 16 NS B bytes of the packed
// row.  W is read once.
//
// Bound by the shared-memory pipe and by issue slots, both at 60 %, with too few warps to hide what depends on what: 26.7
// wavefronts per 32 points (a cell record, 8 random bytes, takes 5.6, the candidate codewords 14: 4 per read from
// eight copies, the fourth only where there is one; rotation shuffles 3) and 106 instructions with the default codebook of
// 2048; 27.5 and 116 with one of 12 updates on 2^15 samples, of whose cells more overflow.  Four layers of 13B with the
// latter: 4.01 ms with 33.7 wavefronts per 32 points, 3.09 ms now.
// QUANT: 0 = nearest codeword through the cell table, 1 = polar quantiser, 2 = no quantiser at all:
// the kernel then is the calibration pass of Section 3.4, which visits n = min(d_out, 1024) rows
// floor(t d_out / n) and adds up the pair moduli |(y_2k, y_2k+1)| per pair position.  The row groups of a
// block add their sums up in shared memory, in ascending order, and every block leaves one slot of partial sums per
// matrix in the workspace; calibrate_finish2_kernel adds the slots in ascending order, so the result does not
// depend on timing.
template <bool BF16, int LOG2B, int NS, int MAXT, int QUANT>
__global__ void __launch_bounds__(MAXT, 1) encode2_kernel(const Encode2Args a) {
    constexpr bool POLAR = QUANT == 1, CALIB = QUANT == 2;
    constexpr int WE = 256 * NS;
    typedef Lay2<NS, LOG2B> Lay;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double ss_part[2][32];  // per-warp partial sums of squares, two rows in flight
    __shared__ MatDesc cur;            // the matrix the block is working on (re-read per row: saves registers)
    __shared__ int used_rows[16];      // calibration: rows that each group has added up
    __shared__ int row_words[2];       // words of a packed row of the matrix: with payload, and up to its stride
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;

    chain_release();
    const int cb_bytes = QUANT != 0 ? 0 : (a.K * 8) << a.log2c;  // only the table search reads codewords
    if (QUANT == 0) fill_codebook_copies(reinterpret_cast<float2*>(smem), a.codebook, a.K, a.log2c);
    unsigned char* table = smem + cb_bytes;
    if (!CALIB) {
        uint4* dst = reinterpret_cast<uint4*>(table);
        const int n16 = a.table_bytes / 16;
        for (int base = 0; base < n16; base += 8 * blockDim.x) {
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = base + u * blockDim.x + threadIdx.x;
                if (i < n16) v[u] = load_blob(a.table + i);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = base + u * blockDim.x + threadIdx.x;
                if (i < n16) dst[i] = v[u];
            }
        }
    }

    SearchSmem s;
    search_fields(s, smem, a.K, a.log2K, a.log2c, 3 + a.log2c);
    s.cells = smem_addr(table) - 8u * kMagicBits * uint32_t(a.grid + 1);
    s.overflow = smem_addr(table + a.off_overflow);
    s.grid = uint32_t(a.grid);
    s.zlo = a.map_zlo;
    s.c0 = a.map_c0;
    s.c1 = a.map_c1;
    s.c2 = a.map_c2;
    s.bias = a.map_bias;
    PolarSmem ps;
    ps.thr2 = smem_addr(table);
    ps.bnd = smem_addr(table + a.off_overflow);
    ps.Ba = a.polar_ba;
    ps.Bp = a.polar_bp;

    const int B = a.log2K;
    constexpr int kEsz = BF16 ? 2 : 4;
    uint32_t first[NS];  // see store_indices
#pragma unroll
    for (int p = 0; p < NS; ++p) {
        const uint32_t bit0 = uint32_t(4 * B * Lay::octet_after(lane, p)), w = (bit0 + 31) >> 5;
        first[p] = w | ((32 * w - bit0) << 16);
    }

    // the span is written once, before the batch handle exists
    const int4 span = block_span(a.spans, CALIB ? min(a.one.d_out, QAMW_CALIB_MAX_ROWS) : a.one.d_out);
    chain_wait();
    for (int m = span.x; m <= span.z; ++m) {
        // The warps regroup when the row length changes: nobody may still be inside the previous
        // matrix (its named barriers and partial sums) when the first warp enters the next one.  The
        // first pass also waits for the tables.  (The first descriptor ahead of the wait: 0.3 us less for one matrix, but the
        // compiler then spills more in the row loop, 3092 -> 3253 us for four layers of 13B.)
        __syncthreads();
        if (threadIdx.x == 0) {
            cur = a.descs ? a.descs[m] : a.one;
            row_words[0] = int((((long long)(cur.d_in >> 1) * B + 7) / 8 + 3) / 4);
            row_words[1] = int(cur.packed_row_stride >> 2);
        }
        __syncthreads();
        const MatDesc& d = cur;
        const int d_in = d.d_in, n_pairs = d_in >> 1;
        const int row_begin = m == span.x ? span.y : 0;
        const int n_cal = min(d.d_out, QAMW_CALIB_MAX_ROWS);  // calibration walks this many rows
        const int row_end = m == span.z ? span.w : (CALIB ? n_cal : d.d_out);
        const int n_seg = (d_in + WE - 1) / WE;
        const int groups = min(15, n_warps / n_seg);  // named barriers 1..15
        const int group = warp / n_seg, seg = warp - group * n_seg;
        const int row0 = group < groups ? row_begin + group : row_end;
        if (!CALIB && row0 >= row_end) continue;
        const int row_step = groups;
        const int tg = n_seg * 32;
        const int oct0 = seg * (WE / 8);

        // The first row is asked for together with the constants where registers are left for it.
        constexpr bool kEarly = MAXT <= 512;
        const int col0 = seg * WE + 8 * NS * lane;  // first column of this thread
        // Raw bits of the thread's elements of one row.  The next row is fetched between the searches of the thread's
        // octets: early enough for its latency to hide, and late enough that its registers are those of the points
        // searched already (with both alive, 72 and 80 registers a thread spilled into the row loop: 58
        // against 46 cycles per 32 points).  Columns beyond the row stay zero.
        constexpr int kRaw = BF16 ? 4 * NS : 8 * NS;
        uint32_t raw[kRaw];
        auto fetch = [&](int t) {
            const long long row = CALIB ? (long long)t * cur.d_out / n_cal : t;
            const char* wp = static_cast<const char*>(cur.W) + (row * cur.w_row_stride + col0) * kEsz;
            if (a.wide) {
                if (col0 < d_in) {
#pragma unroll
                    for (int h = 0; h < kRaw / 8; ++h) {
                        uint32_t w[8];
                        ld_global_256(wp + 32 * h, w);
#pragma unroll
                        for (int i = 0; i < 8; ++i) raw[8 * h + i] = w[i];
                    }
                }
            } else {
#pragma unroll
                for (int h = 0; h < kRaw / 4; ++h)  // 16 bytes: an octet of bf16, half of one of f32
                    if (col0 + 16 * h / kEsz < d_in) {
                        const uint4 w = *reinterpret_cast<const uint4*>(wp + 16 * h);
                        raw[4 * h] = w.x;
                        raw[4 * h + 1] = w.y;
                        raw[4 * h + 2] = w.z;
                        raw[4 * h + 3] = w.w;
                    }
            }
        };
#pragma unroll
        for (int i = 0; i < kRaw; ++i) raw[i] = 0u;
        if (kEarly && row0 < row_end) fetch(row0);
        // per-column constants: t_j = s_j sign_j of the columns the thread loads; reciprocal pair scales
        // (with the butterfly's sign pattern folded in) of the pairs it holds after the rotation
        f32x2 t[NS][4];
        float q[NS][4];
        uint32_t live = 0;  // bit p: the octet that ends up in slot p lies inside the row
        bool risky = false;
        {
            int e_oct[NS], k_oct[NS];
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                e_oct[p] = oct0 + Lay::octet_before(lane, p);
                k_oct[p] = oct0 + Lay::octet_after(lane, p);
            }
            Columns<NS, !CALIB> cols;
            cols.load(d.chan_scale, d.signs, d.sigma, e_oct, k_oct, d_in);
#pragma unroll
            for (int p = 0; p < NS; ++p) {
                float cs[8], sgn[8];
                cols.unpack(p, 8 * e_oct[p] < d_in, cs, sgn);
#pragma unroll
                for (int i = 0; i < 4; ++i) t[p][i] = pack2(cs[2 * i] * sgn[2 * i], cs[2 * i + 1] * sgn[2 * i + 1]);
                const bool in = 8 * k_oct[p] < d_in;
                live |= in ? 1u << p : 0u;
                if (!CALIB) {
                    const float4 v = cols.sg[CALIB ? 0 : p];
                    const float sg[4] = {v.x, v.y, v.z, v.w};
                    const float fl = Lay::negated(lane, p) ? -1.0f : 1.0f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // q_k = f32(1 / (double)sigma_k): the correctly rounded f32 reciprocal is the same number
                        const float r = in ? __frcp_rn(sg[i]) : 0.f;
                        // |z| <= q (1 + eps) because |y| <= 1 for a unit row: only a huge reciprocal pair scale can
                        // carry a point beyond the table's reach
                        risky |= !(r < 15000.0f);
                        q[p][i] = fl * r;
                    }
                }
            }
        }
        if (!kEarly && row0 < row_end) fetch(row0);
        const uint32_t careful = a.brute || __any_sync(kFull, risky) ? 1u : 0u;

        const int seg_word0 = 4 * NS * B * seg;     // first packed word of this warp's segment (16 NS B bytes per segment)
        const bool last_seg = seg == n_seg - 1;
        double* part_base = &ss_part[0][group * n_seg];

        int parity = 0;
        double acc[NS][4];
        int used = 0;
#pragma unroll
        for (int p = 0; p < NS; ++p)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[p][i] = 0.0;
        for (int row = row0; row < row_end; row += row_step, parity ^= 1) {
            f32x2 P[NS][4];
            if (BF16) {
#pragma unroll
                for (int i = 0; i < 4 * NS; ++i)
                    P[i >> 2][i & 3] = mul2(pack2(__uint_as_float(raw[i] << 16), __uint_as_float(raw[i] & 0xffff0000u)),
                                            t[i >> 2][i & 3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4 * NS; ++i)
                    P[i >> 2][i & 3] = mul2(pack2(__uint_as_float(raw[2 * i]), __uint_as_float(raw[2 * i + 1])), t[i >> 2][i & 3]);
            }
            if (CALIB && row + row_step < row_end) fetch(row + row_step);
            // sum of squares of the row: ss = sum_j (double)x_j^2, per thread, per warp, then per row
            double* part = part_base + parity * 32;
            {
                double s0 = 0.0, s1 = 0.0;
#pragma unroll
                for (int p = 0; p < NS; ++p)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float x0, x1;
                        unpack2(P[p][i], x0, x1);
                        const double d0 = double(x0), d1 = double(x1);
                        s0 = fma(d0, d0, s0);
                        s1 = fma(d1, d1, s1);
                    }
                s0 = warp_total(s0 + s1);
                if (lane == 0) part[seg] = s0;
            }
            // The rotation does not need the norm, so the warps of the row meet only after it.  A
            // warp can be one row ahead of another at most, hence the two sets of partial sums.
            fwht2<NS, LOG2B, false>(P, lane, a.log2b);
            group_barrier(group, tg);
            // every warp adds the same numbers in the same order
            const float r = float(sqrt(warp_total(lane < n_seg ? part[lane] : 0.0)));
            // g = f32(c_b / r); 0 for a zero row (all its pairs become the origin) and for a non-finite
            // row (its indices are unspecified; the searches accept any input)
            const float gn = isfinite(r) && r > 0.f ? __fdiv_rn(a.inv_sqrt_b, r) : 0.f;
            if (lane == 0 && seg == 0) {
                if (!CALIB) cur.row_norm[row] = r;
                if (!isfinite(r) && a.status) atomicOr(a.status, 1);
            }
            const f32x2 gn2 = pack2(gn, gn);
            if constexpr (CALIB) {  // calibration: rows of zero (or non-finite) norm are skipped
                if (gn != 0.f) {
                    ++used;
#pragma unroll
                    for (int p = 0; p < NS; ++p)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float y0, y1;
                            unpack2(mul2(P[p][i], gn2), y0, y1);
                            acc[p][i] += double(sqrtf(__fmaf_rn(y1, y1, __fmul_rn(y0, y0))));
                        }
                }
            } else {
                uint2 octet[NS];  // 4 B bits
#pragma unroll
                for (int p = 0; p < NS; ++p) {
                    if (p == NS / 2 && row + row_step < row_end) fetch(row + row_step);
                    uint32_t v[4];
                    float2 z[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float yx, yy;
                        unpack2(mul2(P[p][i], gn2), yx, yy);
                        z[i] = make_float2(__fmul_rn(yx, q[p][i]), __fmul_rn(yy, q[p][i]));
                    }
                    if (POLAR) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[i] = uint32_t(search_polar(ps, z[i].x, z[i].y));
                    } else {
                        uint32_t word1[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[i] = search_cell<false>(s, z[i].x, z[i].y, word1[i]);
                        // one of the four cells has more than four candidates, or points may lie beyond the table
                        if (cell_overflows(word1[0] | word1[1] | word1[2] | word1[3] | careful)) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                if (careful && !(fmaxf(fabsf(z[i].x), fabsf(z[i].y)) < a.reach))
                                    v[i] = search_exhaustive(s, z[i].x, z[i].y);
                                else if (cell_overflows(word1[i]))
                                    v[i] = search_overflow<false>(s, word1[i], first_list_word(s, word1[i]), v[i], z[i].x, z[i].y);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[i] >>= s.log2_entry;
                    }
                    // two indices fit a 32-bit word (B <= 12); octets beyond the row are packed as zero
                    const uint32_t lo = v[0] | (v[1] << B), hi = v[2] | (v[3] << B);
                    const bool in = live & (1u << p);
                    octet[p].x = in ? lo | (2 * B < 32 ? hi << (2 * B) : 0u) : 0u;
                    octet[p].y = in ? hi >> (32 - 2 * B) : 0u;
                }
                uint32_t* out = reinterpret_cast<uint32_t*>(cur.packed + (long long)row * cur.packed_row_stride) + seg_word0;
                const int payload = row_words[0] - seg_word0;
                store_indices<NS, LOG2B>(octet, first, B, out, payload, lane);
                if (last_seg)  // padding up to the row stride is written as zero
                    for (int w = payload + lane; w < row_words[1] - seg_word0; w += 32) out[w] = 0u;
            }  // !CALIB
        }
        if constexpr (CALIB) {
            double* sums = reinterpret_cast<double*>(smem);  // [group][n_pairs]
            if (group < groups) {
#pragma unroll
                for (int p = 0; p < NS; ++p)
                    if (live & (1u << p)) {
                        const int k0 = 4 * (oct0 + Lay::octet_after(lane, p));
#pragma unroll
                        for (int i = 0; i < 4; ++i) sums[group * n_pairs + k0 + i] = acc[p][i];
                    }
                if (lane == 0 && seg == 0) used_rows[group] = used;
            }
            __syncthreads();
            const int pair_stride = (n_pairs + 3) & ~3;
            const int slot = int(blockIdx.x) - cur.calib_first_block;
            double* ws = reinterpret_cast<double*>(a.calib_base + cur.calib_offset);
            for (int k = threadIdx.x; k < n_pairs; k += blockDim.x) {
                double v = 0.0;
                for (int g = 0; g < groups; ++g) v += sums[g * n_pairs + k];
                ws[size_t(slot) * pair_stride + k] = v;
            }
            if (threadIdx.x == 0) {
                int n = 0;
                for (int g = 0; g < groups; ++g) n += used_rows[g];
                ws[size_t(cur.calib_slots) * pair_stride + slot] = double(n);
            }
        }
    }
}

// sigma_k of every matrix from the slots of partial sums, one per block that the matrix was spread over.  A block
// owns 32 pair positions of one matrix; its eight warps each add a contiguous slice of the slots in ascending
// order, and the slice sums are then added in ascending order: the result does not depend on timing.  Bound by the
// latency of its loads, which come in one step.  (Sixteen slices: 1 us less for one matrix, 2 to 10 us more for the batches, whose slots are few.)
constexpr int kFinishSlices = 8;
__global__ void __launch_bounds__(32 * kFinishSlices) calibrate_finish2_kernel(const MatDesc* descs, const MatDesc one,
                                                                             const unsigned char* calib_base) {
    __shared__ double part_sum[kFinishSlices][32], part_used[kFinishSlices];
    chain_release();
    chain_wait();
    const MatDesc& d = descs ? descs[blockIdx.y] : one;
    const int n_pairs = d.d_in >> 1, pair_stride = (n_pairs + 3) & ~3;
    if (int(blockIdx.x) * 32 >= n_pairs) return;
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    const double* ws = reinterpret_cast<const double*>(calib_base + d.calib_offset);
    const int per = (d.calib_slots + kFinishSlices - 1) / kFinishSlices;
    const int s0 = min(d.calib_slots, slice * per), s1 = min(d.calib_slots, s0 + per);
    double sum = 0.0, used = 0.0;
    for (int slot = s0 + lane; slot < s1; slot += 32) used += ws[size_t(d.calib_slots) * pair_stride + slot];  // whole numbers: any order
    if (k < n_pairs) {
        constexpr int U = 20;  // a slot per SM: one step
        for (int slot = s0; slot < s1; slot += U) {
            double v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = slot + u < s1 ? ws[size_t(slot + u) * pair_stride + k] : 0.0;
#pragma unroll
            for (int u = 0; u < U; ++u) sum += v[u];
        }
    }
    used = warp_total(used);
    part_sum[slice][lane] = sum;
    if (lane == 0) part_used[slice] = used;
    __syncthreads();
    if (slice == 0 && k < n_pairs) {
        double s = 0.0, u = 0.0;
        for (int i = 0; i < kFinishSlices; ++i) {
            s += part_sum[i][lane];
            u += part_used[i];
        }
        const double inv_sqrt_d = 1.0 / sqrt(double(d.d_in));
        double sg = u > 0.0 ? (s / u) / sqrt(1.5707963267948966) : inv_sqrt_d;  // Rayleigh mean = sigma sqrt(pi / 2)
        sg = fmax(sg, 1e-4 * inv_sqrt_d);
        const_cast<float*>(d.sigma)[k] = float(sg);
    }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
inline bool aligned(const void* p, uintptr_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; }

int launch_check(const char* what, cudaError_t e) {
    if (e != cudaSuccess) {
        set_cuda_error(what, int(e));
        return QAMW_ERR_CUDA;
    }
    return QAMW_OK;
}

// cudaFuncSetAttribute once per kernel and device (the call is not free and the value never changes)
int raise_smem_limit(const void* kernel) {
    static std::mutex mu;
    static std::unordered_map<const void*, unsigned long long> done;  // kernel -> bit mask of devices
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    std::lock_guard<std::mutex> lock(mu);
    unsigned long long& mask = done[kernel];
    if (mask & bit) return QAMW_OK;
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess)  // the limit covers static and dynamic shared memory together
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemLimit - fa.sharedSizeBytes));
    if (e != cudaSuccess) {
        set_cuda_error("cudaFuncSetAttribute", int(e));
        return QAMW_ERR_NOMEM;
    }
    mask |= bit;
    return QAMW_OK;
}

template <int LOG2B>
int launch_decode2(const Decode2Args& a, bool fits, int blocks, int threads, size_t smem, cudaStream_t st) {
    auto kernel = fits ? decode2_kernel<LOG2B, true> : decode2_kernel<LOG2B, false>;
    int rc = raise_smem_limit(reinterpret_cast<const void*>(kernel));
    if (rc) return rc;
    return launch_check("decode2_kernel", launch_chained(kernel, blocks, threads, smem, st, a));
}

template <bool BF16, int LOG2B, int NS, int MAXT>
int launch_encode2(const Encode2Args& a, int blocks, int threads, size_t smem, cudaStream_t st) {
    if (a.calib_base) {
        int rc = raise_smem_limit(reinterpret_cast<const void*>(&encode2_kernel<BF16, LOG2B, NS, MAXT, 2>));
        if (rc) return rc;
        return launch_check("encode2_kernel (calibrate)",
                            launch_chained(encode2_kernel<BF16, LOG2B, NS, MAXT, 2>, blocks, threads, smem, st, a));
    }
    if constexpr (LOG2B >= 5 && LOG2B <= 9) if (a.polar_ba >= 0) {
        int rc = raise_smem_limit(reinterpret_cast<const void*>(&encode2_kernel<BF16, LOG2B, NS, MAXT, 1>));
        if (rc) return rc;
        return launch_check("encode2_kernel (polar)",
                            launch_chained(encode2_kernel<BF16, LOG2B, NS, MAXT, 1>, blocks, threads, smem, st, a));
    }
    int rc = raise_smem_limit(reinterpret_cast<const void*>(&encode2_kernel<BF16, LOG2B, NS, MAXT, 0>));
    if (rc) return rc;
    return launch_check("encode2_kernel", launch_chained(encode2_kernel<BF16, LOG2B, NS, MAXT, 0>, blocks, threads, smem, st, a));
}

constexpr size_t kEncode2StaticSmem = 1024;  // ss_part and the current matrix descriptor, rounded up

}  // namespace

namespace qamw {

// Contiguous spans of the concatenated row list, one per block, of (nearly) equal cost.  A block works
// on `groups` rows at a time, each row step taking about the same time whatever the row length, so
// a row of matrix i costs 1 / groups_i: row_cost[i] = lcm / groups_i in integer units.
void make_spans(const MatDesc* descs, int n, int n_blocks, const int* row_cost, std::vector<int4>* out) {
    std::vector<long long> cum(n + 1, 0);
    for (int i = 0; i < n; ++i) cum[i + 1] = cum[i] + (long long)descs[i].d_out * row_cost[i];
    const long long total = cum[n];
    auto locate = [&](long long pos, int* m, int* row) {  // first row that starts at or after cost position `pos`
        int i = int(std::upper_bound(cum.begin(), cum.end(), pos) - cum.begin()) - 1;
        i = std::min(std::max(i, 0), n - 1);
        const long long r = (pos - cum[i] + row_cost[i] - 1) / row_cost[i];
        *m = i;
        *row = int(std::min<long long>(r, descs[i].d_out));
    };
    out->resize(n_blocks);
    int m0 = 0, r0 = 0;
    for (int k = 0; k < n_blocks; ++k) {
        int m1, r1;
        if (k == n_blocks - 1) {
            m1 = n - 1;
            r1 = descs[n - 1].d_out;
        } else {
            locate(total / n_blocks * (k + 1) + (total % n_blocks) * (k + 1) / n_blocks, &m1, &r1);
        }
        (*out)[k] = make_int4(m0, r0, m1, r1);
        m0 = m1;
        r0 = r1;
    }
}

int rows_decode(const MatDesc* descs_dev, const MatDesc* descs_host, int n, const void* spans_dev, int span_blocks,
                int block, int K, const float* codebook_dev, uint32_t flags, void* stream, int* count) {
    constexpr int NS = kDecodeSlots, WE = 256 * NS, kWarps = kDecodeWarps;
    const int log2b = ilog2(block);
    if (n <= 0) return QAMW_ERR_SHAPE;
    long long pairs = 0;
    bool fits = true;
    for (int i = 0; i < n; ++i) {
        const MatDesc& d = descs_host[i];
        if (d.d_in % 8 || d.d_in > WE * kWarps) return QAMW_ERR_SHAPE;
        if (!aligned(d.w_hat, 16) || !aligned(d.packed, 16) || d.packed_row_stride % 4) return QAMW_ERR_SHAPE;
        if (!aligned(d.chan_scale, 16) || !aligned(d.signs, 8) || !aligned(d.sigma, 16)) return QAMW_ERR_SHAPE;
        fits = fits && aligned(d.w_hat, 32) && d.d_in % 16 == 0 && d.packed_row_stride % 16 == 0;
        pairs += (long long)d.d_out * (d.d_in / 2);
    }
    if (pairs == 0) return QAMW_OK;
    int grid = sm_count();
    if (flags & QAMW_FLAG_HALF_DEVICE) grid = std::max(1, grid / 2);
    // A single matrix is spread over all SMs before a block gets a second row, so a small one runs with few warps
    // per block and few codebook copies.
    int warps = kWarps, blocks = span_blocks;
    if (!spans_dev) {
        const int n_seg = (descs_host[0].d_in + WE - 1) / WE;
        const int groups = std::max(1, std::min(kWarps / n_seg, (descs_host[0].d_out + grid - 1) / grid));
        warps = groups * n_seg;
        blocks = std::max(1, std::min(grid, (descs_host[0].d_out + groups - 1) / groups));
    }
    Decode2Args a;
    a.descs = descs_dev;
    a.one = descs_host[0];
    a.spans = static_cast<const int4*>(spans_dev);
    a.codebook = reinterpret_cast<const float2*>(codebook_dev);
    a.K = K;
    a.log2K = ilog2(K);
    a.seg_bytes = 16 * NS * a.log2K;
    a.stage_bytes = (a.seg_bytes + 28 + 127) & ~127;  // 12 bytes before a row off its boundary, 16 read past its end
    a.log2b = log2b;
    a.inv_sqrt_b = float(1.0 / std::sqrt(double(block)));
    const size_t stage_total = size_t(warps) * kDecodeDepth * a.stage_bytes;
    a.log2c = pick_copies(K, pairs / 32 / blocks, std::min(size_t(128) * 1024, kSmemLimit - stage_total));
    const size_t smem = (size_t(K) * 8 << a.log2c) + stage_total;
    if (count) {
        ++*count;
        return QAMW_OK;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = QAMW_ERR_SHAPE;
    switch (log2b >= 5 ? log2b : 0) {
        case 0: rc = launch_decode2<0>(a, fits, blocks, warps * 32, smem, st); break;
        case 5: rc = launch_decode2<5>(a, fits, blocks, warps * 32, smem, st); break;
        case 6: rc = launch_decode2<6>(a, fits, blocks, warps * 32, smem, st); break;
        case 7: rc = launch_decode2<7>(a, fits, blocks, warps * 32, smem, st); break;
        case 8: rc = launch_decode2<8>(a, fits, blocks, warps * 32, smem, st); break;
        case 9: rc = launch_decode2<9>(a, fits, blocks, warps * 32, smem, st); break;
        case 10: rc = launch_decode2<10>(a, fits, blocks, warps * 32, smem, st); break;
        default: break;
    }
    return rc;
}

// Block sizes of the encoder: 16, 20, 24 or 28 warps.  The register file is split over the four
// schedulers of an SM, 16384 registers each, so 4, 5, 6 or 7 warps per scheduler leave 128, 96, 80 or 72
// registers per thread.  With all warps busy the sizes take 45.9, 47.6, 51.2 and 49.4 us for 8192 rows of 2048 (fewer
// registers, less of a row's search in flight; the last two spill a little), and time grows with the share of warps
// that a row length leaves idle (whole groups of n_seg warps, at most 15 groups): the size with the
// largest product of the two is taken; 0 if the row is too long.
// Hadamard blocks of 1024 elements need all 32 lanes with four octets each: 16 warps.
int encode_groups(int warps, int n_seg) { return std::min(15, warps / n_seg); }
int encode_segment(int block) { return block == 1024 ? 1024 : 512; }
constexpr int kEncodeClasses = 4;
constexpr int kEncodeWarps[kEncodeClasses] = {16, 20, 24, 28};
int encode_warps(int n_seg, int block) {
    if (block == 1024) return n_seg <= 16 ? 16 : 0;
    const double full[kEncodeClasses] = {1.0, 45.9 / 47.6, 45.9 / 51.2, 45.9 / 49.4};
    int best = 0;
    double best_rate = 0.0;
    for (int c = 0; c < kEncodeClasses; ++c) {
        const double rate = full[c] * encode_groups(kEncodeWarps[c], n_seg) * n_seg / kEncodeWarps[c];
        if (rate > best_rate) {
            best = kEncodeWarps[c];
            best_rate = rate;
        }
    }
    return best;
}
int encode_class(int warps) {  // rows too long for any size end up in the last class and fall back later
    return warps ? (warps - 16) / 4 : kEncodeClasses - 1;
}
int decode_groups(int n_seg) { return kDecodeWarps / n_seg; }
constexpr int kCostUnit = 360360;  // divisible by every group count 1..15

int rows_encode(const MatDesc* descs_dev, const MatDesc* descs_host, int n, const void* spans_dev, int span_blocks,
                int block, int K, int w_bf16, const ::qamw_codebook* cb, uint32_t flags, int32_t* status, void* stream,
                void* calib_base, int* count) {
    const int log2b = ilog2(block), WE = encode_segment(block), NS = WE / 256;
    if (n <= 0) return QAMW_ERR_SHAPE;
    const size_t esz = w_bf16 ? 2 : 4;
    int max_seg = 1, warps = 0;
    long long rows = 0;
    bool wide = true;
    for (int i = 0; i < n; ++i) {
        const MatDesc& d = descs_host[i];
        if (d.d_in % 8) return QAMW_ERR_SHAPE;
        const size_t row_bytes = size_t(d.w_row_stride) * esz;
        if (!aligned(d.W, 16) || row_bytes % 16) return QAMW_ERR_SHAPE;
        wide = wide && aligned(d.W, 32) && row_bytes % 32 == 0 && d.d_in % (8 * NS) == 0;
        if (!aligned(d.chan_scale, 16) || !aligned(d.signs, 8) || (!calib_base && !aligned(d.sigma, 16))) return QAMW_ERR_SHAPE;
        const int n_seg = (d.d_in + WE - 1) / WE;
        max_seg = std::max(max_seg, n_seg);
        warps = std::max(warps, encode_warps(n_seg, block));
        rows += calib_base ? std::min(d.d_out, QAMW_CALIB_MAX_ROWS) : d.d_out;
    }
    if (max_seg > warps) return QAMW_ERR_SHAPE;  // also: a row too long for any block size
    // the polar quantiser is built for the layouts of the models it is compared on
    if (!calib_base && cb->polar && (log2b < 5 || log2b > 9 || !wide)) return QAMW_ERR_SHAPE;
    if (rows == 0) return QAMW_OK;
    Encode2Args a;
    a.descs = descs_dev;
    a.one = descs_host[0];
    a.spans = static_cast<const int4*>(spans_dev);
    a.calib_base = static_cast<unsigned char*>(calib_base);
    const bool calib = calib_base != nullptr;
    a.codebook = calib ? nullptr : static_cast<const float2*>(cb->d_blob);
    a.table = calib ? nullptr : reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(cb->d_blob) + cb->off_cells);
    a.table_bytes = calib ? 0 : int(cb->blob_bytes - cb->off_cells);
    a.off_overflow = calib ? 0 : int(cb->off_overflow - cb->off_cells);
    a.K = K;
    a.log2K = ilog2(K);
    a.grid = calib ? 1 : cb->map.grid;
    auto twice = [](float v) {
        uint32_t bits;
        std::memcpy(&bits, &v, 4);
        return (f32x2(bits) << 32) | bits;
    };
    a.map_zlo = twice(calib ? 0.f : -cb->map.zmax);
    a.map_c0 = twice(calib ? 0.f : cb->map.c0);
    a.map_c1 = twice(calib ? 0.f : cb->map.c1);
    a.map_c2 = twice(calib ? 0.f : cb->map.c2);
    a.map_bias = twice(calib ? 0.f : 12582912.0f + float(cb->map.half));
    a.log2b = log2b;
    a.wide = wide;
    a.brute = (flags & QAMW_FLAG_BRUTE_FORCE) ? 1 : 0;
    a.reach = a.brute ? -1.0f : 16000.0f;
    a.inv_sqrt_b = float(1.0 / std::sqrt(double(block)));
    a.status = status;
    const bool polar = !calib && cb->polar;
    a.polar_ba = polar ? cb->polar_ba : -1;
    a.polar_bp = polar ? cb->polar_bp : -1;
    const bool tables = !calib && !polar;
    a.log2c = tables ? cb->log2c : 0;
    // calibration: the block's groups meet in shared memory, a double per pair of every warp's segment
    const size_t smem = calib ? size_t(warps) * (WE / 2) * sizeof(double)
                              : ((size_t(a.table_bytes) + 15) & ~size_t(15)) + (tables ? size_t(K) * 8 << a.log2c : 0);
    if (smem > kSmemLimit - kEncode2StaticSmem) return QAMW_ERR_SHAPE;
    int grid = sm_count();
    if (flags & QAMW_FLAG_HALF_DEVICE) grid = std::max(1, grid / 2);
    int blocks = spans_dev ? span_blocks : int(std::max<long long>(1, std::min<long long>(grid, rows)));
    if (!spans_dev && calib) blocks = descs_host[0].calib_slots;
    if (count) {
        ++*count;
        return QAMW_OK;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = QAMW_ERR_SHAPE;
#define QAMW_ENC2(LB)                                                                          \
    case LB:                                                                                   \
        if (warps == 28)                                                                       \
            rc = w_bf16 ? launch_encode2<true, LB, 2, 896>(a, blocks, 896, smem, st)           \
                        : launch_encode2<false, LB, 2, 896>(a, blocks, 896, smem, st);         \
        else if (warps == 24)                                                                  \
            rc = w_bf16 ? launch_encode2<true, LB, 2, 768>(a, blocks, 768, smem, st)           \
                        : launch_encode2<false, LB, 2, 768>(a, blocks, 768, smem, st);         \
        else if (warps == 20)                                                                  \
            rc = w_bf16 ? launch_encode2<true, LB, 2, 640>(a, blocks, 640, smem, st)           \
                        : launch_encode2<false, LB, 2, 640>(a, blocks, 640, smem, st);         \
        else                                                                                   \
            rc = w_bf16 ? launch_encode2<true, LB, 2, 512>(a, blocks, 512, smem, st)           \
                        : launch_encode2<false, LB, 2, 512>(a, blocks, 512, smem, st);         \
        break;
    switch (log2b >= 5 ? log2b : 0) {
        QAMW_ENC2(0)
        QAMW_ENC2(5)
        QAMW_ENC2(6)
        QAMW_ENC2(7)
        QAMW_ENC2(8)
        QAMW_ENC2(9)
        case 10:
            rc = w_bf16 ? launch_encode2<true, 10, 4, 512>(a, blocks, 512, smem, st)
                        : launch_encode2<false, 10, 4, 512>(a, blocks, 512, smem, st);
            break;
        default: break;
    }
#undef QAMW_ENC2
    return rc;
}

int rows_calibrate(MatDesc d, int block, int w_bf16, uint32_t flags, void* workspace, size_t workspace_bytes, int32_t* status,
                   void* stream) {
    const int n_rows = std::min(d.d_out, QAMW_CALIB_MAX_ROWS);
    if (n_rows == 0) return QAMW_ERR_SHAPE;
    // as many blocks as have a row for each of their groups: every one leaves a slot for the finish to add up
    const int WE = encode_segment(block), n_seg = (d.d_in + WE - 1) / WE, warps = encode_warps(n_seg, block);
    if (!warps) return QAMW_ERR_SHAPE;
    int grid = sm_count();
    if (flags & QAMW_FLAG_HALF_DEVICE) grid = std::max(1, grid / 2);
    const int groups = encode_groups(warps, n_seg);
    const size_t slot = (size_t((d.d_in / 2 + 3) & ~3) + 1) * sizeof(double);
    d.calib_offset = 0;
    d.calib_first_block = 0;
    d.calib_slots = int(std::min<size_t>(size_t(std::min(grid, (n_rows + groups - 1) / groups)), workspace_bytes / slot));
    if (d.calib_slots < 1) return QAMW_ERR_SHAPE;
    const int rc = rows_encode(nullptr, &d, 1, nullptr, 0, block, 2, w_bf16, nullptr, flags, status, stream, workspace);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return launch_check("calibrate_finish2_kernel",
                        launch_chained(calibrate_finish2_kernel, dim3(unsigned((d.d_in / 2 + 31) / 32)), 32 * kFinishSlices, 0, st,
                                       nullptr, d, static_cast<unsigned char*>(workspace)));
}

}  // namespace qamw

// ---------------------------------------------------------------------------------------------
// batches: all linear weights of a layer or a model behind one handle
// ---------------------------------------------------------------------------------------------
// A set of matrices that one launch of a row kernel walks: their descriptors on the device and one
// span of the concatenated row list per block.
struct RowSet {
    std::vector<int> index;         // positions in the batch
    std::vector<MatDesc> descs;     // host copy of the device array
    MatDesc* d_descs = nullptr;
    int4* d_spans = nullptr;
};

struct qamw_batch {
    int n = 0;
    int device = -1;
    int block = 0, K = 0, w_dtype = 0;
    const qamw_codebook* cb = nullptr;
    std::vector<qamw_matrix> items;
    int n_blocks = 0;
    RowSet dec;                     // all matrices, spans weighted for the decoder's geometry
    RowSet enc[kEncodeClasses];     // encoder: one set per block size
    int4* d_spans_dist = nullptr;   // distortion: spans of the concatenated work-item list, over dec.d_descs
    int n_blocks_dist = 0;
    double* d_dist_partial = nullptr;   // one record of four sums per (block, matrix of its span)
    DistOwner* d_dist_owner = nullptr;  // per matrix: first and last block whose span holds it, first record
    unsigned int* d_dist_counter = nullptr;  // tickets of the blocks, per matrix; zero between launches
    MatDesc* d_cal_all = nullptr;       // calibration descriptors of all block-size classes, for the one finish launch
    int cal_all_n = 0, cal_all_max_pairs = 0;
    RowSet cal[kEncodeClasses];     // calibration: the encoder's sets again, spans over the calibration rows
    size_t cal_bytes = 0;           // partial-sum slots of all matrices (front of the caller's workspace)
    std::vector<size_t> ws_offset;  // calibration scratch of item i inside the caller's workspace
    size_t ws_bytes = 0;
};

namespace {
MatDesc make_desc(const qamw_matrix& it) {
    MatDesc d{};
    d.W = it.W;
    d.chan_scale = it.chan_scale;
    d.signs = it.signs;
    d.sigma = it.sigma;
    d.act_rms = it.act_rms;
    d.packed = it.packed;
    d.row_norm = it.row_norm;
    d.w_hat = it.w_hat_bf16;
    d.dist4 = it.dist4;
    d.w_row_stride = it.p.w_row_stride;
    d.packed_row_stride = it.p.packed_row_stride;
    d.d_out = it.p.d_out;
    d.d_in = it.p.d_in;
    return d;
}
}  // namespace

namespace {
void free_row_set(RowSet& r) {
    if (r.d_descs) cudaFree(r.d_descs);
    if (r.d_spans) cudaFree(r.d_spans);
    r.d_descs = nullptr;
    r.d_spans = nullptr;
}
cudaError_t upload_row_set(RowSet& r, int n_blocks, const std::vector<int>& row_cost) {
    if (r.descs.empty()) return cudaSuccess;
    std::vector<int4> spans;
    make_spans(r.descs.data(), int(r.descs.size()), n_blocks, row_cost.data(), &spans);
    cudaError_t e = cudaMalloc(&r.d_descs, sizeof(MatDesc) * r.descs.size());
    if (e == cudaSuccess) e = cudaMemcpy(r.d_descs, r.descs.data(), sizeof(MatDesc) * r.descs.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&r.d_spans, sizeof(int4) * spans.size());
    if (e == cudaSuccess) e = cudaMemcpy(r.d_spans, spans.data(), sizeof(int4) * spans.size(), cudaMemcpyHostToDevice);
    return e;
}
}  // namespace

extern "C" int qamw_batch_create(const qamw_matrix* items, int n, const qamw_codebook* cb, qamw_batch** out) {
    if (!items || n <= 0 || !cb || !out) return QAMW_ERR_ARG;
    *out = nullptr;
    for (int i = 0; i < n; ++i) {
        int rc = check_matrix_params(&items[i].p);
        if (rc) return rc;
        const qamw_params& p = items[i].p;
        if (p.block != items[0].p.block || p.K != items[0].p.K || p.w_dtype != items[0].p.w_dtype) return QAMW_ERR_ARG;
        if (p.K != cb->K || !items[i].signs) return QAMW_ERR_ARG;
        const size_t row_bytes = qamw_packed_row_bytes(p.d_in, p.K);
        if (p.packed_row_stride < (long long)row_bytes || p.packed_row_stride % 4) return QAMW_ERR_ALIGN;
        if (reinterpret_cast<uintptr_t>(items[i].packed) % 4) return QAMW_ERR_ALIGN;
    }
    int device = -1;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) {
        set_cuda_error("qamw_batch_create", int(e));
        return QAMW_ERR_CUDA;
    }
    if (device != cb->device) return QAMW_ERR_ARG;  // the codebook lives on another device
    qamw_batch* b = new (std::nothrow) qamw_batch();
    if (!b) return QAMW_ERR_NOMEM;
    b->n = n;
    b->device = device;
    b->block = items[0].p.block;
    b->K = items[0].p.K;
    b->w_dtype = items[0].p.w_dtype;
    b->cb = cb;
    b->items.assign(items, items + n);
    b->n_blocks = sm_count();
    std::vector<int> dec_cost, enc_cost[kEncodeClasses];
    for (int i = 0; i < n; ++i) {
        const MatDesc d = make_desc(items[i]);
        b->ws_offset.push_back(b->ws_bytes);
        b->ws_bytes += (qamw_calibrate_workspace_bytes(&items[i].p) + 255) & ~size_t(255);
        const int seg4 = (d.d_in + 1023) / 1024, seg2 = (d.d_in + encode_segment(b->block) - 1) / encode_segment(b->block);
        b->dec.index.push_back(i);
        b->dec.descs.push_back(d);
        dec_cost.push_back(kCostUnit / std::max(1, decode_groups(std::min(seg4, 16))));
        const int warps = encode_warps(seg2, b->block);
        const int c = encode_class(warps);
        b->enc[c].index.push_back(i);
        b->enc[c].descs.push_back(d);
        enc_cost[c].push_back(kCostUnit / std::max(1, encode_groups(warps ? warps : 28, std::min(seg2, 28))));
    }
    e = upload_row_set(b->dec, b->n_blocks, dec_cost);
    for (int c = 0; c < kEncodeClasses && e == cudaSuccess; ++c) e = upload_row_set(b->enc[c], b->n_blocks, enc_cost[c]);
    for (int c = 0; c < kEncodeClasses && e == cudaSuccess; ++c) {  // calibration: min(d_out, 1024) rows per matrix
        RowSet& r = b->cal[c];
        r.index = b->enc[c].index;
        r.descs = b->enc[c].descs;
        if (r.descs.empty()) continue;
        const int m = int(r.descs.size());
        std::vector<MatDesc> cal_rows(r.descs);
        for (MatDesc& d : cal_rows) d.d_out = std::min(d.d_out, QAMW_CALIB_MAX_ROWS);
        std::vector<int4> spans;
        make_spans(cal_rows.data(), m, b->n_blocks, enc_cost[c].data(), &spans);
        std::vector<int> first(size_t(m), b->n_blocks), last(size_t(m), -1);
        for (int k = 0; k < b->n_blocks; ++k)
            for (int i = spans[size_t(k)].x; i <= spans[size_t(k)].z; ++i) {
                first[size_t(i)] = std::min(first[size_t(i)], k);
                last[size_t(i)] = std::max(last[size_t(i)], k);
            }
        for (int i = 0; i < m; ++i) {
            MatDesc& d = r.descs[size_t(i)];
            d.calib_first_block = first[size_t(i)];
            d.calib_slots = std::max(0, last[size_t(i)] - first[size_t(i)] + 1);
            d.calib_offset = (long long)b->cal_bytes;
            const size_t pair_stride = (size_t(d.d_in / 2) + 3) & ~size_t(3);
            b->cal_bytes += ((size_t(d.calib_slots) * (pair_stride + 1)) * sizeof(double) + 255) & ~size_t(255);
        }
        e = cudaMalloc(&r.d_descs, sizeof(MatDesc) * size_t(m));
        if (e == cudaSuccess) e = cudaMemcpy(r.d_descs, r.descs.data(), sizeof(MatDesc) * size_t(m), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMalloc(&r.d_spans, sizeof(int4) * spans.size());
        if (e == cudaSuccess) e = cudaMemcpy(r.d_spans, spans.data(), sizeof(int4) * spans.size(), cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) {  // all calibration descriptors in one array: one finish launch for every class
        std::vector<MatDesc> all;
        for (int c = 0; c < kEncodeClasses; ++c) all.insert(all.end(), b->cal[c].descs.begin(), b->cal[c].descs.end());
        b->cal_all_n = int(all.size());
        for (const MatDesc& d : all) b->cal_all_max_pairs = std::max(b->cal_all_max_pairs, d.d_in / 2);
        if (!all.empty()) {
            e = cudaMalloc(&b->d_cal_all, sizeof(MatDesc) * all.size());
            if (e == cudaSuccess) e = cudaMemcpy(b->d_cal_all, all.data(), sizeof(MatDesc) * all.size(), cudaMemcpyHostToDevice);
        }
    }
    // Distortion: equal numbers of work items per block.  Five blocks fit an SM, one wave.  bf16 rows run through a ring that
    // a block fills and drains once: with few items one wave is best, with many more and shorter blocks even out what the
    // SMs lose to each other.  us with 5, 16 and 24 blocks per SM, by items per block of one wave: 3.7 (a layer of 1.1B)
    // 40.0, 45.9, 43.6; 14.9 (four of them) 137.9, 140.0, 137.4; 16.8 (a layer of 7B) 157.3, 157.6, 154.9; 26.4 (13B) 241,
    // 238, 237; 33.6 306, 301, 285; 105 (four layers of 13B) 974, 909, 886; 1055 (forty) 10114, 9322, 9197.  f32 rows
    // have no ring and lose what a last partial wave leaves idle: 58.8, 74.9, 66.3 at 3.7; 349, 408, 379 at 26.4; 1365,
    // 1579, 1409 at 105.  bf16 rows off 16 bytes have none either, and 5 and 24 blocks do alike: 209, 224, 214 at 15.3;
    // 404, 438, 405 at 30.6; 1596, 1686, 1545 at 122.
    if (e == cudaSuccess) {
        std::vector<MatDesc> items_as_rows(b->dec.descs);
        std::vector<int> unit(size_t(n), 1);
        long long total = 0;
        for (int i = 0; i < n; ++i) {
            items_as_rows[size_t(i)].d_out = int(distortion_items(b->dec.descs[size_t(i)].d_out, b->dec.descs[size_t(i)].d_in));
            total += items_as_rows[size_t(i)].d_out;
        }
        const long long wave = 5LL * b->n_blocks;
        const bool many = b->w_dtype == QAMW_DTYPE_BF16 && total >= 20 * wave;
        b->n_blocks_dist = int(std::max<long long>(1, std::min<long long>(many ? 24LL * b->n_blocks : wave, total)));
        std::vector<int4> spans;
        make_spans(items_as_rows.data(), n, b->n_blocks_dist, unit.data(), &spans);
        e = cudaMalloc(&b->d_spans_dist, sizeof(int4) * spans.size());
        if (e == cudaSuccess) e = cudaMemcpy(b->d_spans_dist, spans.data(), sizeof(int4) * spans.size(), cudaMemcpyHostToDevice);
        // per matrix: the blocks whose span holds it and where their records go
        std::vector<DistOwner> owner(size_t(n), DistOwner{int(spans.size()), -1, 0});
        for (size_t k = 0; k < spans.size(); ++k)
            for (int i = spans[k].x; i <= spans[k].z; ++i) {
                owner[size_t(i)].first = std::min(owner[size_t(i)].first, int(k));
                owner[size_t(i)].last = std::max(owner[size_t(i)].last, int(k));
            }
        int n_rec = 0;
        for (int i = 0; i < n; ++i) {
            owner[size_t(i)].offset = n_rec;
            n_rec += std::max(0, owner[size_t(i)].last - owner[size_t(i)].first + 1);
        }
        if (e == cudaSuccess) e = cudaMalloc(&b->d_dist_partial, sizeof(double) * 4 * size_t(std::max(1, n_rec)));
        if (e == cudaSuccess) e = cudaMalloc(&b->d_dist_owner, sizeof(DistOwner) * size_t(n));
        if (e == cudaSuccess) e = cudaMemcpy(b->d_dist_owner, owner.data(), sizeof(DistOwner) * size_t(n), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMalloc(&b->d_dist_counter, sizeof(unsigned int) * size_t(n));
        if (e == cudaSuccess) e = cudaMemset(b->d_dist_counter, 0, sizeof(unsigned int) * size_t(n));
    }
    // the handle may be used on a stream that does not wait for the default one
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        set_cuda_error("qamw_batch_create", int(e));
        qamw_batch_destroy(b);
        return QAMW_ERR_CUDA;
    }
    *out = b;
    return QAMW_OK;
}

extern "C" void qamw_batch_destroy(qamw_batch* b) {
    if (!b) return;
    free_row_set(b->dec);
    for (int c = 0; c < kEncodeClasses; ++c) {
        free_row_set(b->enc[c]);
        free_row_set(b->cal[c]);
    }
    if (b->d_spans_dist) cudaFree(b->d_spans_dist);
    if (b->d_dist_partial) cudaFree(b->d_dist_partial);
    if (b->d_dist_owner) cudaFree(b->d_dist_owner);
    if (b->d_dist_counter) cudaFree(b->d_dist_counter);
    if (b->d_cal_all) cudaFree(b->d_cal_all);
    delete b;
}

// The front of the workspace holds the slots of the batched pass, the rest the scratch of the
// single-matrix calls that matrices outside the common layout fall back to.
extern "C" size_t qamw_batch_workspace_bytes(const qamw_batch* b) { return b ? b->cal_bytes + b->ws_bytes : 0; }

extern "C" int qamw_calibrate_batch(const qamw_batch* b, void* workspace, size_t workspace_bytes, int32_t* status_out,
                                    void* stream) {
    if (!b || !workspace) return QAMW_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(workspace) % 8) return QAMW_ERR_ALIGN;
    if (workspace_bytes < b->cal_bytes + b->ws_bytes) return QAMW_ERR_NOMEM;
    for (int i = 0; i < b->n; ++i)
        if (!b->items[i].W || !b->items[i].sigma) return QAMW_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t flags = b->items[0].p.flags;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    // One pass per block size; the partial sums of all of them are finished by one launch, unless a class
    // had to go through the single-matrix kernels (then the classes that did not are finished one by one).
    bool fast[kEncodeClasses] = {}, any_fast = false, any_general = false;
    for (int c = 0; c < kEncodeClasses; ++c) {
        const RowSet& set = b->cal[c];
        if (set.descs.empty()) continue;
        int rc = QAMW_ERR_SHAPE;
        if (!(flags & QAMW_FLAG_GENERAL_KERNELS)) {
            rc = rows_encode(set.d_descs, set.descs.data(), int(set.descs.size()), set.d_spans, b->n_blocks, b->block, b->K,
                             b->w_dtype == QAMW_DTYPE_BF16, nullptr, flags, status_out, stream, ws);
            fast[c] = rc == QAMW_OK;
            any_fast = any_fast || fast[c];
        }
        if (rc == QAMW_ERR_SHAPE) {  // some matrix of the set needs the general kernel: one call per matrix
            any_general = true;
            rc = QAMW_OK;
            for (size_t k = 0; k < set.index.size() && rc == QAMW_OK; ++k) {
                const int i = set.index[k];
                const qamw_matrix& it = b->items[i];
                rc = qamw_calibrate(it.W, &it.p, it.chan_scale, it.signs, it.sigma, ws + b->cal_bytes + b->ws_offset[i],
                                    workspace_bytes - b->cal_bytes - b->ws_offset[i], status_out, stream);
            }
        }
        if (rc) return rc;
    }
    if (!any_general && any_fast) {
        return launch_check("calibrate_finish2_kernel",
                            launch_chained(calibrate_finish2_kernel, dim3(unsigned((b->cal_all_max_pairs + 31) / 32), unsigned(b->cal_all_n)),
                                           32 * kFinishSlices, 0, st, b->d_cal_all, MatDesc{}, ws));
    }
    for (int c = 0; c < kEncodeClasses; ++c) {
        if (!fast[c]) continue;
        const RowSet& set = b->cal[c];
        int max_pairs = 0;
        for (const MatDesc& d : set.descs) max_pairs = std::max(max_pairs, d.d_in / 2);
        const int rc = launch_check("calibrate_finish2_kernel",
                                    launch_chained(calibrate_finish2_kernel, dim3(unsigned((max_pairs + 31) / 32), unsigned(set.descs.size())),
                                                   32 * kFinishSlices, 0, st, set.d_descs, MatDesc{}, ws));
        if (rc) return rc;
    }
    return QAMW_OK;
}

extern "C" int qamw_encode_batch(const qamw_batch* b, int32_t* status_out, void* stream) {
    if (!b) return QAMW_ERR_ARG;
    for (int i = 0; i < b->n; ++i) {
        const qamw_matrix& it = b->items[i];
        if (!it.W || !it.sigma || !it.packed || !it.row_norm) return QAMW_ERR_ARG;
    }
    const uint32_t flags = b->items[0].p.flags;
    for (int c = 0; c < kEncodeClasses; ++c) {  // one launch per block size
        const RowSet& set = b->enc[c];
        if (set.descs.empty()) continue;
        int rc = QAMW_ERR_SHAPE;
        if (!(flags & QAMW_FLAG_GENERAL_KERNELS))
            rc = rows_encode(set.d_descs, set.descs.data(), int(set.descs.size()), set.d_spans, b->n_blocks, b->block, b->K,
                             b->w_dtype == QAMW_DTYPE_BF16, b->cb, flags, status_out, stream);
        if (rc == QAMW_ERR_SHAPE) {  // some matrix of the class needs the general kernel: one call per matrix
            rc = QAMW_OK;
            for (size_t k = 0; k < set.index.size() && rc == QAMW_OK; ++k) {
                const qamw_matrix& it = b->items[set.index[k]];
                rc = qamw_encode(it.W, &it.p, it.chan_scale, it.signs, it.sigma, b->cb, it.packed, it.row_norm, status_out,
                                 stream);
            }
        }
        if (rc) return rc;
    }
    return QAMW_OK;
}

extern "C" int qamw_decode_batch(const qamw_batch* b, void* stream) {
    if (!b) return QAMW_ERR_ARG;
    for (int i = 0; i < b->n; ++i) {
        const qamw_matrix& it = b->items[i];
        if (!it.sigma || !it.packed || !it.row_norm || !it.w_hat_bf16) return QAMW_ERR_ARG;
    }
    const uint32_t flags = b->items[0].p.flags;
    int rc = QAMW_ERR_SHAPE;
    if (!(flags & QAMW_FLAG_GENERAL_KERNELS))
        rc = rows_decode(b->dec.d_descs, b->dec.descs.data(), b->n, b->dec.d_spans, b->n_blocks, b->block, b->K,
                         static_cast<const float*>(b->cb->d_blob), flags, stream);
    if (rc != QAMW_ERR_SHAPE) return rc;
    for (int i = 0; i < b->n; ++i) {  // some matrix needs the general kernel: one call per matrix
        const qamw_matrix& it = b->items[i];
        rc = qamw_decode(it.packed, it.row_norm, it.chan_scale, it.signs, it.sigma, b->cb, &it.p, it.w_hat_bf16, stream);
        if (rc) return rc;
    }
    return QAMW_OK;
}

extern "C" int qamw_distortion_batch(const qamw_batch* b, void* stream) {
    if (!b) return QAMW_ERR_ARG;
    for (int i = 0; i < b->n; ++i) {
        const qamw_matrix& it = b->items[i];
        if (!it.W || !it.w_hat_bf16 || !it.dist4) return QAMW_ERR_ARG;
    }
    DistReduce red;
    red.partial = b->d_dist_partial;
    red.owner = b->d_dist_owner;
    red.counter = b->d_dist_counter;
    return distortion_batch_launch(b->dec.d_descs, b->d_spans_dist, b->n_blocks_dist, b->w_dtype == QAMW_DTYPE_BF16,
                                   red, stream);
}

// Kernels that the four phases launch, by the rules that they launch them by.
extern "C" int qamw_batch_launches(const qamw_batch* b, int32_t* per_phase_out) {
    if (!b) return QAMW_ERR_ARG;
    const uint32_t flags = b->items[0].p.flags;
    const bool general = flags & QAMW_FLAG_GENERAL_KERNELS, bf16 = b->w_dtype == QAMW_DTYPE_BF16;
    int passes = 0, single = 0, encode = 0, decode = 0;
    char any = 0;  // stands for the workspace, which a counted call does not touch
    for (int c = 0; c < kEncodeClasses; ++c) {
        const RowSet &cal = b->cal[c], &enc = b->enc[c];
        const int n = int(enc.descs.size());
        if (n == 0) continue;
        if (general || rows_encode(cal.d_descs, cal.descs.data(), n, cal.d_spans, b->n_blocks, b->block, b->K, bf16, nullptr, flags,
                                   nullptr, nullptr, &any, &passes))
            single += n;
        if (general || rows_encode(enc.d_descs, enc.descs.data(), n, enc.d_spans, b->n_blocks, b->block, b->K, bf16, b->cb, flags,
                                   nullptr, nullptr, nullptr, &encode))
            for (const MatDesc& d : enc.descs) encode += d.d_out > 0;
    }
    const int calibrate = passes + 2 * single + (single ? passes : passes > 0);  // one finish for all classes, or one each
    if (general || rows_decode(b->dec.d_descs, b->dec.descs.data(), b->n, b->dec.d_spans, b->n_blocks, b->block, b->K, nullptr, flags,
                               nullptr, &decode))
        for (const MatDesc& d : b->dec.descs) decode += d.d_out > 0;
    const int phases[4] = {calibrate, encode, decode, 1};
    if (per_phase_out) std::copy(phases, phases + 4, per_phase_out);
    return phases[0] + phases[1] + phases[2] + phases[3];
}
