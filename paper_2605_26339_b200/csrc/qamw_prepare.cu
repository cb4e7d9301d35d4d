// Channel scales and sign mask on the device, for the one-call quantiser.  The activation statistics arrive in the
// kernel's own parameters: the host neither computes logarithms (40 us at 4096 channels, 12 at 1024) nor queues copies,
// which would break the chain of kernels on the stream.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cstring>

#include "qamw_device.cuh"
#include "qamw_internal.h"
#include "qamw_launch.h"

using namespace qamw;
namespace cg = cooperative_groups;

namespace {

constexpr int kPrepBlocks = 8, kPrepThreads = 256;  // one cluster; 512 threads take 0.5 us longer at 1024 channels
constexpr int kPrepMaxPerThread = 16384 / (kPrepBlocks * kPrepThreads);

struct PrepArgs {
    const float* act;   // NULL: in the parameters
    float* chan_scale;  // NULL: signs only
    int8_t* signs;
    uint64_t seed;
    float alpha;
    int d_in;
};
template <int N>
struct PrepParams {
    PrepArgs a;
    float act[N];
};

// s_j = clamp(exp(alpha log r_j - mean), 1/16, 16) in double, as qamw_channel_scales; signs as qamw_make_signs.
// Everything but the stores comes before the wait when the statistics are in the parameters: what follows the wait is on the
// critical path of a chain of kernels that last two to five microseconds each.
template <int N>
__global__ void __cluster_dims__(kPrepBlocks) __launch_bounds__(kPrepThreads) prepare_kernel(const __grid_constant__ PrepParams<N> p) {
    __shared__ double part[kPrepThreads / 32], block_sum;
    const PrepArgs& a = p.a;
    cg::cluster_group cluster = cg::this_cluster();
    const int j0 = blockIdx.x * kPrepThreads + threadIdx.x;
    constexpr int kStep = kPrepBlocks * kPrepThreads;
    chain_release();
    if (a.act) chain_wait();  // the kernel before this one has written them
    double t[kPrepMaxPerThread], sum = 0.0;
#pragma unroll
    for (int i = 0; i < kPrepMaxPerThread; ++i) {
        const int j = j0 + i * kStep;
        t[i] = 0.0;
        if (j >= a.d_in) break;
        if (!a.chan_scale) continue;
        double r = double(a.act ? a.act[j] : p.act[j < N ? j : 0]);
        if (!(r > double(FLT_MIN))) r = double(FLT_MIN);
        t[i] = double(a.alpha) * log(r);
        sum += t[i];
    }
    auto store_signs = [&]() {
        for (int j = j0; j < a.d_in; j += kStep) a.signs[j] = column_sign(a.seed, j);
    };
    if (!a.chan_scale) {  // the same for all blocks
        chain_wait();
        store_signs();
        return;
    }
    sum = warp_sum(sum);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kPrepThreads / 32; ++w) s += part[w];
        block_sum = s;
    }
    cluster.sync();
    double mean = 0.0;
    for (int b = 0; b < kPrepBlocks; ++b) mean += *cluster.map_shared_rank(&block_sum, b);
    mean /= double(a.d_in);
    cluster.sync();  // nobody leaves while its sum is still read
    float s[kPrepMaxPerThread];
#pragma unroll
    for (int i = 0; i < kPrepMaxPerThread; ++i) {
        s[i] = 0.f;
        if (j0 + i * kStep >= a.d_in) break;
        s[i] = float(fmin(16.0, fmax(1.0 / 16.0, exp(t[i] - mean))));
    }
    if (!a.act) chain_wait();
    store_signs();
#pragma unroll
    for (int i = 0; i < kPrepMaxPerThread; ++i) {
        const int j = j0 + i * kStep;
        if (j >= a.d_in) break;
        a.chan_scale[j] = s[i];
    }
}

// Statistics of a row too long for one kernel's parameters, piece by piece, to where the scales will be.
template <int N>
__global__ void __launch_bounds__(kPrepThreads) upload_kernel(const __grid_constant__ PrepParams<N> p, int first, int n) {
    chain_release();
    chain_wait();
    const int i = blockIdx.x * kPrepThreads + threadIdx.x;
    if (i < n) p.a.chan_scale[first + i] = p.act[i];
}

template <int N>
cudaError_t launch_prepare(const PrepArgs& a, const float* act_host, cudaStream_t st) {
    PrepParams<N> p;
    p.a = a;
    if (!act_host || a.d_in <= N) {
        if (act_host) std::memcpy(p.act, act_host, size_t(a.d_in) * sizeof(float));
        return launch_chained(prepare_kernel<N>, kPrepBlocks, kPrepThreads, 0, st, p);
    }
    for (int first = 0; first < a.d_in; first += N) {
        const int n = std::min(N, a.d_in - first);
        std::memcpy(p.act, act_host + first, size_t(n) * sizeof(float));
        const cudaError_t e = launch_chained(upload_kernel<N>, (n + kPrepThreads - 1) / kPrepThreads, kPrepThreads, 0, st, p, first, n);
        if (e != cudaSuccess) return e;
    }
    p.a.act = a.chan_scale;
    return launch_chained(prepare_kernel<N>, kPrepBlocks, kPrepThreads, 0, st, p);
}

}  // namespace

namespace qamw {

int prepare_columns(const float* act_host, int d_in, float alpha, uint64_t seed, float* chan_scale, int8_t* signs, void* stream) {
    PrepArgs a{};
    a.chan_scale = act_host ? chan_scale : nullptr;
    a.signs = signs;
    a.seed = seed;
    a.alpha = alpha;
    a.d_in = d_in;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // a kernel takes at most 32764 bytes of parameters; short rows do not send a long one's
    const cudaError_t e = !act_host || d_in <= 1024 ? launch_prepare<1024>(a, act_host, st)
                          : d_in <= 2048            ? launch_prepare<2048>(a, act_host, st)
                          : d_in <= 4096            ? launch_prepare<4096>(a, act_host, st)
                                                    : launch_prepare<8064>(a, act_host, st);
    if (e != cudaSuccess) {
        set_cuda_error("prepare_kernel", int(e));
        return QAMW_ERR_CUDA;
    }
    return QAMW_OK;
}

}  // namespace qamw
