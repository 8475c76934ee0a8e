// Noise-floor normalisation and per-SFT noise weights: the step before the
// F-statistic path for coloured, non-stationary noise (the paper's client
// assumes white SFTs; the weighted multi-detector sum is the reading of
// Listing 1's per-detector sum and normalized(result) used here).
//
//   P_k   = Re^2 + Im^2 in FP32 (squares rounded, then the sum rounded)
//   S(k)  = median{P_j : |j - k| <= W, j stored} / ln 2, FP32, computed as
//           (m1 + m2) * 0.5 / ln 2 with m1, m2 the two middle values (equal
//           for an odd count; the window is clipped at the band edges)
//   X'_k  = X_k / sqrt(S(k))   (0 where S(k) = 0)
//   w     = (1 / Sbar) / mean over SFTs of (1 / Sbar), Sbar = mean_k S(k)
//           (0 where Sbar = 0, left out of the mean), FP64
//
// The median is selected by stable ranks in the window, which picks exactly the
// elements a sort would, so S matches an FP32 reference bit for bit.
#include <limits>

#include "fstat_internal.cuh"

namespace fs {
namespace {

constexpr float kLn2f = 0.69314718055994530942f;
constexpr int kNoiseBlock = 256;

// Floors S of bins k0 .. k1-1 of one SFT, by a warp.  The lanes hold the window
// (slot = lane + 32 r, NR <= 5 a lane) with each value's stable rank in it
// (smaller values, then equal ones further left).  A step to the next bin puts
// the incoming value into the outgoing one's slot and moves the ranks of the
// values above either; so a bin costs O(window) instead of the O(window^2) of
// counting every rank afresh.  A slot outside the band holds NaN, which compares
// false, and a rank that no median has.
template <int NR>
__device__ __forceinline__ void sliding_floor(const float* pw, int n_bins, int half, int k0, int k1, float* floor) {
    const int lane = threadIdx.x & 31, m = 2 * half + 1;
    const float nan = std::numeric_limits<float>::quiet_NaN();
    constexpr int kNone = -(1 << 24);
    float v[NR];
    int rank[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int slot = lane + 32 * r, j = k0 - half + slot;
        v[r] = slot < m && j >= 0 && j < n_bins ? pw[j] : nan;
        rank[r] = v[r] == v[r] ? 0 : kNone;
    }
    for (int j = max(0, k0 - half); j <= min(n_bins - 1, k0 + half); ++j) {
        const float x = pw[j];
#pragma unroll
        for (int r = 0; r < NR; ++r) rank[r] += (x < v[r]) || (x == v[r] && j < k0 - half + lane + 32 * r);
    }
    int slot = 0;
    float mine = 0.f;   // floor of the bin k0 + 32 i + lane
    for (int k = k0; k < k1; ++k) {
        const int n = min(n_bins - 1, k + half) - max(0, k - half) + 1;
        const int r1 = (n - 1) >> 1, r2 = n >> 1;   // equal for an odd count
        auto pick = [&](int want) {
            float x = 0.f;
            bool has = false;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const bool is = rank[r] == want;
                x = is ? v[r] : x;
                has |= is;
            }
            return __shfl_sync(0xffffffffu, x, __ffs(__ballot_sync(0xffffffffu, has)) - 1);
        };
        const float m1 = pick(r1), m2 = r1 == r2 ? m1 : pick(r2);
        const int at = (k - k0) & 31;
        if (lane == at) mine = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
        if (at == 31 || k + 1 == k1)
            if (lane <= at) floor[k - at + lane] = __fdiv_rn(mine, kLn2f);
        // on to k + 1
        const int jo = k - half, ji = k + 1 + half;
        const float out = jo >= 0 ? pw[jo] : nan, in = ji < n_bins ? pw[ji] : nan;
        int below = out <= in ? -1 : 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            below += __popc(__ballot_sync(0xffffffffu, v[r] <= in));
            rank[r] += (v[r] > in ? 1 : 0) - (out <= v[r] ? 1 : 0);
        }
        below = in == in ? below : kNone;
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (slot == lane + 32 * r) {
                v[r] = in;
                rank[r] = below;
            }
        slot = slot + 1 == m ? 0 : slot + 1;
    }
}

// One block per SFT: powers into shared memory, the running medians (each warp
// a run of bins), then per bin the whitened bin, and the SFT's mean floor.
// Bound: instruction issue of the medians, about 30 + 14 NR a bin and warp.
// 2400 SFTs x 1816 bins, half width 32: 472 us against 3820 us with every rank
// counted afresh.
template <int NR>
__global__ void __launch_bounds__(kNoiseBlock) noise_floor_kernel(const float2* __restrict__ bins, long long row,
                                                                 int n_bins, int half, float* floor,
                                                                 float2* __restrict__ white,
                                                                 double* __restrict__ sbar) {
    extern __shared__ float pw[];   // [n_bins]
    __shared__ double red[kNoiseBlock / 32];
    const int s = blockIdx.x;
    const float2* x = bins + (size_t)s * row;
    for (int k = threadIdx.x; k < n_bins; k += blockDim.x) {
        const float2 v = x[k];
        pw[k] = __fadd_rn(__fmul_rn(v.x, v.x), __fmul_rn(v.y, v.y));
    }
    __syncthreads();
    constexpr int kWarps = kNoiseBlock / 32;
    const int run = (n_bins + kWarps - 1) / kWarps, k0 = ((int)threadIdx.x >> 5) * run;
    float* fl = floor + (size_t)s * n_bins;
    if (k0 < n_bins) sliding_floor<NR>(pw, n_bins, half, k0, min(n_bins, k0 + run), fl);
    __syncthreads();
    double acc = 0.0;
    for (int k = threadIdx.x; k < n_bins; k += blockDim.x) {
        const float S = fl[k];
        acc += (double)S;
        const float2 v = x[k];
        float2 o = make_float2(0.f, 0.f);
        if (S > 0.f) {
            const float inv = __fdiv_rn(1.0f, __fsqrt_rn(S));
            o = make_float2(v.x * inv, v.y * inv);
        }
        white[(size_t)s * row + k] = o;
    }
    for (long long k = n_bins + threadIdx.x; k < row; k += blockDim.x) white[(size_t)s * row + k] = make_float2(0.f, 0.f);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kNoiseBlock / 32; ++w) t += red[w];
        sbar[s] = t / (double)n_bins;
    }
}

// Weights from the mean floors of all SFTs (one block).
__global__ void __launch_bounds__(kNoiseBlock) noise_weight_kernel(const double* __restrict__ sbar, int n_sft,
                                                                  double* __restrict__ weight) {
    __shared__ double rs[kNoiseBlock / 32];
    __shared__ int rc[kNoiseBlock / 32];
    double sum = 0.0;
    int cnt = 0;
    for (int i = threadIdx.x; i < n_sft; i += blockDim.x)
        if (sbar[i] > 0.0) {
            sum += 1.0 / sbar[i];
            ++cnt;
        }
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if ((threadIdx.x & 31) == 0) {
        rs[threadIdx.x >> 5] = sum;
        rc[threadIdx.x >> 5] = cnt;
    }
    __syncthreads();
    __shared__ double mean;
    if (threadIdx.x == 0) {
        double t = 0.0;
        int c = 0;
        for (int w = 0; w < kNoiseBlock / 32; ++w) {
            t += rs[w];
            c += rc[w];
        }
        mean = c > 0 ? t / (double)c : 1.0;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_sft; i += blockDim.x) weight[i] = sbar[i] > 0.0 ? (1.0 / sbar[i]) / mean : 0.0;
}

}  // namespace

cudaError_t launch_noise_floor(const float2* bins, long long row, int n_sft, int n_bins, int half, float* floor,
                               float2* white, double* sbar, double* weight, cudaStream_t s) {
    const size_t smem = (size_t)n_bins * sizeof(float);
    auto launch = [&](auto kernel) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kernel<<<n_sft, kNoiseBlock, smem, s>>>(bins, row, n_bins, half, floor, white, sbar);
        return cudaGetLastError();
    };
    const int nr = (2 * half + 1 + 31) / 32;   // half <= 64
    const cudaError_t e = nr <= 1   ? launch(noise_floor_kernel<1>)
                          : nr == 2 ? launch(noise_floor_kernel<2>)
                          : nr == 3 ? launch(noise_floor_kernel<3>)
                          : nr == 4 ? launch(noise_floor_kernel<4>)
                                    : launch(noise_floor_kernel<5>);
    if (e != cudaSuccess) return e;
    noise_weight_kernel<<<1, kNoiseBlock, 0, s>>>(sbar, n_sft, weight);
    return cudaGetLastError();
}

}  // namespace fs
