// Toplist: the K largest 2F of a bank, ordered by (2F descending, template
// index ascending).  2F >= 0, so the FP32 bit patterns order like the values.
//
// The values are read once.  They are cut into G <= 32768 groups of
// consecutive values; the K-th largest group maximum is a lower bound of the
// K-th largest value (K groups hold one such value each), and every value that
// can be in the list lies in a group whose maximum reaches it.  So:
//   group_max  the maximum of every group, and a histogram of the maxima;
//   pivot      the K-th largest maximum, to 22 bits, rounded down;
//   gather     the values >= pivot of the groups that reach it (K groups or a
//              few more, about K values: with K << G few groups hold two);
//   rank       each candidate's place is the number of candidates before it,
//              counted directly; places < K are written out.
// Candidates come in any order, ranks do not depend on it: the result is
// deterministic.  Where more values reach the pivot than the candidate buffer
// holds (mostly equal or sorted values), the five kernels of an exact
// three-level radix select over all values (11 + 11 + 10 bits) run before
// rank; otherwise they return at once (1.7 us each).  Up to kDirect
// values, rank alone runs on the values.
//
// Bound: reading the values (HBM) for large banks, group_max at 6.4 TB/s; the
// launches for small ones.  Whole list, against a radix select with one-thread
// scans of its histograms and five passes over the values: 60 M values, K = 1000
// 96 us (586 before); 1.8 M 55 us (152); 800 values, K = 20 11 us (168).  All
// values equal, 60 M: 426 us (549).
#include "fstat_internal.cuh"

#include <algorithm>
#include <cstdio>
#include <mutex>

#include "../../include/fstat_noalloc.h"

namespace fs {
namespace {

constexpr int kBins = 2048;
constexpr int kBlk = 256;
constexpr int kGroups = 32768;   // groups at most
constexpr int kCand = 20480;     // candidates at most; a list takes up to 16384
constexpr int kDirect = 8192;    // values ranked without grouping: 25 us for 4096, 44 for 8192; grouped 44 to 88
constexpr int kTieBlocks = 1024;

// Scratch of one toplist (w.scratch), word offsets.  The words before kKeyAt
// start at zero.
// state: [2] threshold bits, [3] count above the threshold,
// [4] ties needed, [5] pivot, [6] candidates, [7] slots taken by collect,
// [8 + 2L], [9 + 2L] prefix and rank of radix level L.
constexpr size_t kStateAt = 0, kHistAt = 16;              // 3 x kBins: radix levels
constexpr size_t kMaxAt = kHistAt + 3 * kBins;            // histogram of the maxima
constexpr size_t kKeyAt = kMaxAt + kBins;
constexpr size_t kTieAt = kKeyAt + kGroups;
constexpr size_t kValAt = kTieAt + kTieBlocks;
constexpr size_t kIdxAt = kValAt + kCand;                 // 64-bit
static_assert(kIdxAt % 2 == 0 && kKeyAt % 4 == 0 && kValAt % 4 == 0, "alignment of the scratch sections");
static_assert((kIdxAt + 2 * kCand) * sizeof(unsigned int) <= kTopkScratch, "scratch of one toplist");

__device__ __forceinline__ void warp_hist_add(unsigned int* h, unsigned int bin, bool valid) {
    const unsigned int act = __ballot_sync(0xffffffffu, valid);
    if (!valid) return;
    const unsigned int peers = __match_any_sync(act, bin);
    const int leader = __ffs(peers) - 1;
    if ((int)(threadIdx.x & 31) == leader) atomicAdd(&h[bin], (unsigned int)__popc(peers));
}

// Ranking key of a value: its FP32 bit pattern, with -0.0 taken as +0.0 (for
// the non-negative values ranked here the patterns order like the values).
__device__ __forceinline__ unsigned int key_bits(float x) {
    const unsigned int b = __float_as_uint(x);
    return b == 0x80000000u ? 0u : b;
}

template <int LEVEL>
__device__ __forceinline__ void classify(unsigned int b, unsigned int prefix, unsigned int& bin, bool& ok) {
    if (LEVEL == 0) {
        bin = b >> 21;
        ok = true;
    } else if (LEVEL == 1) {
        bin = (b >> 10) & 2047u;
        ok = (b >> 21) == prefix;
    } else {
        bin = b & 1023u;
        ok = (b >> 10) == prefix;
    }
}

// Values v[0 .. n-1] as groups of 2^shift (>= 4) from the 16-byte boundary at or
// below v: lead = values of the first group that lie before v.
struct Grouped {
    const float* v;
    long long n;
    int lead, shift, groups;
};

// The four values at position p (a multiple of 4 from that boundary) as keys;
// bit c of `in`: value c exists.  Partial quads are read value by value.
__device__ __forceinline__ uint4 quad(const Grouped& g, long long p, unsigned int& in) {
    const long long i = p - g.lead;
    uint4 k = make_uint4(0u, 0u, 0u, 0u);
    if (i >= 0 && i + 4 <= g.n) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(g.v + i));
        k = make_uint4(key_bits(x.x), key_bits(x.y), key_bits(x.z), key_bits(x.w));
        in = 15u;
        return k;
    }
    unsigned int* kp = &k.x;
    in = 0u;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (i + c >= 0 && i + c < g.n) {
            kp[c] = key_bits(g.v[i + c]);
            in |= 1u << c;
        }
    return k;
}

// A warp takes 2^shift >= 128 values as one group, or 32 quads as several; eight
// quads a lane in flight at full size.  At most 2048 blocks, whose count the
// hardware balances (304 persistent ones: 64 us on 60 M values, 7 rounds for 6.03).
__global__ void __launch_bounds__(512, 2) group_max_kernel(Grouped g, unsigned int* __restrict__ w) {
    __shared__ unsigned int h[kBins];
    for (int i = threadIdx.x; i < kBins; i += 512) h[i] = 0;
    __syncthreads();
    unsigned int* keys = w + kKeyAt;
    const int lane = threadIdx.x & 31;
    const int span = max(g.shift, 7);               // values of a warp: 2^span
    const int width = min(32, 1 << (g.shift - 2));  // lanes of a group
    const long long t = (long long)blockIdx.x * 16 + (threadIdx.x >> 5);
    const long long p0 = (t << span) + 4 * lane, p1 = (t + 1) << span;
    unsigned int m = 0;
    if ((t > 0 || g.lead == 0) && p1 <= g.lead + g.n) {   // all quads whole
        const float4* x4 = reinterpret_cast<const float4*>(g.v + (p0 - g.lead));
        const int quads = 1 << (span - 7);
#pragma unroll 1
        for (int q = 0; q < quads; q += 8) {
            float4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (q + u < quads) x[u] = __ldg(x4 + 32 * (q + u));
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (q + u < quads)
                    m = max(max(m, max(key_bits(x[u].x), key_bits(x[u].y))), max(key_bits(x[u].z), key_bits(x[u].w)));
        }
    } else {
        for (long long p = p0; p < p1; p += 128) {
            unsigned int in;
            const uint4 k = quad(g, p, in);
            m = max(max(m, max(k.x, k.y)), max(k.z, k.w));
        }
    }
    for (int o = 1; o < width; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const long long gi = p0 >> g.shift;
    if ((lane & (width - 1)) == 0 && gi < g.groups) {
        keys[gi] = m;
        atomicAdd(&h[m >> 21], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += 512)
        if (h[i]) atomicAdd(&w[kMaxAt + i], h[i]);
}

// The bin of a kBins-bin histogram that holds the need-th entry from the top,
// and its rank inside that bin; the same in all T threads.  The total is at
// least `need`.
template <int T>
__device__ __forceinline__ uint2 find_bin(const unsigned int* h, unsigned int need) {
    constexpr int kPer = kBins / T;
    __shared__ unsigned int ws[32];
    __shared__ uint2 found;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int top = kBins - 1 - kPer * (int)threadIdx.x;
    unsigned int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        c[i] = h[top - i];
        sum += c[i];
    }
    unsigned int inc = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (threadIdx.x == 0) found = make_uint2(0u, 1u);
    if (lane == 31) ws[warp] = inc;
    __syncthreads();
    unsigned int above = inc - sum;
    for (int i = 0; i < warp; ++i) above += ws[i];
    if (above < need && need <= above + sum) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            if (above < need && need <= above + c[i]) found = make_uint2((unsigned int)(top - i), need - above);
            above += c[i];
        }
    }
    __syncthreads();
    const uint2 r = found;
    __syncthreads();
    return r;
}

// Pivot: the k-th largest maximum with its low 10 bits cleared; 0 if there are
// no k groups.  One block: the maxima's top 11 bits are already counted, the
// next 11 are counted here for the bin that holds the k-th.
__global__ void __launch_bounds__(1024) pivot_kernel(unsigned int* __restrict__ w, int groups, unsigned int k) {
    __shared__ unsigned int h[kBins];
    if ((unsigned int)groups < k) return;   // state[5] is zero
    for (int i = threadIdx.x; i < kBins; i += 1024) h[i] = 0;
    const uint2 a = find_bin<1024>(w + kMaxAt, k);
    const uint4* keys = reinterpret_cast<const uint4*>(w + kKeyAt);
    auto add = [&](unsigned int x, int i) {
        if (i < groups && (x >> 21) == a.x) atomicAdd(&h[(x >> 10) & 2047u], 1u);
    };
#pragma unroll 8
    for (int q = threadIdx.x; 4 * q < groups; q += 1024) {   // the section is a whole number of quads
        const uint4 x = keys[q];
        add(x.x, 4 * q);
        add(x.y, 4 * q + 1);
        add(x.z, 4 * q + 2);
        add(x.w, 4 * q + 3);
    }
    __syncthreads();
    const uint2 b = find_bin<1024>(h, a.y);
    if (threadIdx.x == 0) w[kStateAt + 5] = a.x << 21 | b.x << 10;
}

// Values >= pivot of the groups that reach it.  A block takes consecutive
// groups; its warps share the pieces (512 values, four quads a lane in flight)
// of those that reach the pivot, about K in all.  The count goes on past the end
// of the buffer, which tells the kernels after it.
__global__ void __launch_bounds__(kBlk) gather_kernel(Grouped g, unsigned int* w) {
    __shared__ int hot[kBlk], n_hot;
    const unsigned int pivot = w[kStateAt + 5];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long* idx = reinterpret_cast<long long*>(w + kIdxAt);
    const int per = (g.groups + gridDim.x - 1) / gridDim.x;
    const int g0 = blockIdx.x * per, g1 = min(g.groups, g0 + per);
    const int pshift = max(0, g.shift - 9);   // pieces of a group
    for (int base = g0; base < g1; base += kBlk) {
        __syncthreads();
        if (threadIdx.x == 0) n_hot = 0;
        __syncthreads();
        const int mine = base + (int)threadIdx.x;
        if (mine < g1 && w[kKeyAt + mine] >= pivot) hot[atomicAdd(&n_hot, 1)] = mine;
        __syncthreads();
        const long long pieces = (long long)n_hot << pshift;
        for (long long q = warp; q < pieces; q += kBlk / 32) {
            const long long p0 = ((long long)hot[q >> pshift] << g.shift) + ((q & ((1LL << pshift) - 1)) << 9) + 4 * lane;
            const int size = min(512, 1 << min(g.shift, 9));
            uint4 k[4];
            unsigned int in[4], any = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                in[u] = 0;
                k[u] = make_uint4(0u, 0u, 0u, 0u);
                if (128 * u + 4 * lane < size) k[u] = quad(g, p0 + 128 * u, in[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                in[u] &= (k[u].x >= pivot ? 1u : 0u) | (k[u].y >= pivot ? 2u : 0u) | (k[u].z >= pivot ? 4u : 0u) |
                         (k[u].w >= pivot ? 8u : 0u);
                any += __popc(in[u]);
            }
            if (!__any_sync(0xffffffffu, any != 0)) continue;
            unsigned int off = any;   // inclusive prefix over the lanes
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned int x = __shfl_up_sync(0xffffffffu, off, d);
                if (lane >= d) off += x;
            }
            unsigned int slot = 0;
            if (lane == 31) slot = atomicAdd(&w[kStateAt + 6], off);
            slot = __shfl_sync(0xffffffffu, slot, 31);
            if (slot > (unsigned int)kCand) break;   // overflown: the radix select takes over
            slot += off - any;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned int ks[4] = {k[u].x, k[u].y, k[u].z, k[u].w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (in[u] >> c & 1u) {
                        if (slot < (unsigned int)kCand) {
                            w[kValAt + slot] = ks[c];
                            idx[slot] = p0 + 128 * u + c - g.lead;
                        }
                        ++slot;
                    }
            }
        }
    }
}

// ---- exact radix select, run where the candidates overflow ---------------------------
__device__ __forceinline__ bool overflown(const unsigned int* w) { return w[kStateAt + 6] > (unsigned int)kCand; }

// Bucket of the K-th value at LEVEL, from the histogram of that level: prefix
// and rank inside it, the same in all blocks; block 0 keeps them.
template <int LEVEL>
__device__ __forceinline__ uint2 select_level(unsigned int* w, unsigned int k) {
    if constexpr (LEVEL < 0) {
        return make_uint2(0u, k);
    } else {
        uint2 up = make_uint2(0u, k);
        if constexpr (LEVEL > 0) up = make_uint2(w[kStateAt + 6 + 2 * LEVEL], w[kStateAt + 7 + 2 * LEVEL]);
        const uint2 b = find_bin<kBlk>(w + kHistAt + LEVEL * kBins, up.y);
        const uint2 r = make_uint2(up.x << (LEVEL == 2 ? 10 : 11) | b.x, b.y);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            w[kStateAt + 2 * LEVEL + 8] = r.x;
            w[kStateAt + 2 * LEVEL + 9] = r.y;
        }
        return r;
    }
}

template <int LEVEL>
__global__ void __launch_bounds__(kBlk) hist_kernel(Grouped g, unsigned int* __restrict__ w, unsigned int k) {
    if (!overflown(w)) return;
    __shared__ unsigned int h[kBins];
    for (int i = threadIdx.x; i < kBins; i += kBlk) h[i] = 0;
    const unsigned int prefix = select_level<LEVEL - 1>(w, k).x;
    __syncthreads();
    const long long quads = (g.lead + g.n + 3) >> 2, stride = (long long)gridDim.x * kBlk;
    // every thread of a warp runs the same number of iterations (ballot below)
    for (long long base = (long long)blockIdx.x * kBlk; base < quads; base += stride) {
        unsigned int in = 0;
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (base + threadIdx.x < quads) x = quad(g, 4 * (base + threadIdx.x), in);
        const unsigned int xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            unsigned int bin;
            bool ok;
            classify<LEVEL>(xs[c], prefix, bin, ok);
            warp_hist_add(h, bin, ok && (in >> c & 1u));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += kBlk)
        if (h[i]) atomicAdd(&w[kHistAt + LEVEL * kBins + i], h[i]);
}

// Values above the threshold, in any order, and each block's count of equal ones.
__global__ void __launch_bounds__(kBlk) collect_kernel(const float* __restrict__ v, long long n, long long per_block,
                                                       unsigned int* __restrict__ w, unsigned int k) {
    if (!overflown(w)) return;
    __shared__ unsigned int ties;
    if (threadIdx.x == 0) ties = 0;
    const uint2 last = select_level<2>(w, k);   // threshold, equal values needed
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        w[kStateAt + 2] = last.x;
        w[kStateAt + 3] = k - last.y;
        w[kStateAt + 4] = last.y;
    }
    __syncthreads();
    const unsigned int tau = last.x;
    long long* idx = reinterpret_cast<long long*>(w + kIdxAt);
    const long long lo = (long long)blockIdx.x * per_block;
    const long long hi = min(n, lo + per_block);
    unsigned int my_ties = 0;
    for (long long i = lo + threadIdx.x; i < hi; i += kBlk) {
        const unsigned int b = key_bits(v[i]);
        if (b > tau) {
            const unsigned int s = atomicAdd(&w[kStateAt + 7], 1u);
            idx[s] = i;
            w[kValAt + s] = b;
        } else if (b == tau) {
            ++my_ties;
        }
    }
    for (int o = 16; o > 0; o >>= 1) my_ties += __shfl_xor_sync(0xffffffffu, my_ties, o);
    if ((threadIdx.x & 31) == 0 && my_ties) atomicAdd(&ties, my_ties);
    __syncthreads();
    if (threadIdx.x == 0) w[kTieAt + blockIdx.x] = ties;
}

// The values equal to the threshold that are still needed, in index order.
__global__ void __launch_bounds__(kBlk) tie_kernel(const float* __restrict__ v, long long n, long long per_block,
                                                   unsigned int* __restrict__ w) {
    if (!overflown(w)) return;
    __shared__ unsigned int wsum[kBlk / 32];
    __shared__ unsigned int s_prefix;
    const unsigned int tau = w[kStateAt + 2];
    const unsigned int n_gt = w[kStateAt + 3];
    const unsigned int need = w[kStateAt + 4];
    if (threadIdx.x == 0) s_prefix = 0;
    __syncthreads();
    unsigned int pre = 0;
    for (unsigned int b = threadIdx.x; b < blockIdx.x; b += kBlk) pre += w[kTieAt + b];
    for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(0xffffffffu, pre, o);
    if ((threadIdx.x & 31) == 0 && pre) atomicAdd(&s_prefix, pre);
    __syncthreads();
    unsigned int prefix = s_prefix;
    if (prefix >= need || w[kTieAt + blockIdx.x] == 0) return;
    long long* idx = reinterpret_cast<long long*>(w + kIdxAt);
    const long long lo = (long long)blockIdx.x * per_block;
    const long long hi = min(n, lo + per_block);
    const int wp = threadIdx.x >> 5, l = threadIdx.x & 31;
    for (long long base = lo; base < hi && prefix < need; base += kBlk) {
        const long long i = base + threadIdx.x;
        const bool t = (i < hi) && (key_bits(v[i]) == tau);
        const unsigned int bal = __ballot_sync(0xffffffffu, t);
        if (l == 0) wsum[wp] = __popc(bal);
        __syncthreads();
        unsigned int before = 0, total = 0;
        for (int q = 0; q < kBlk / 32; ++q) {
            if (q < wp) before += wsum[q];
            total += wsum[q];
        }
        const unsigned int rank = prefix + before + __popc(bal & ((1u << l) - 1u));
        if (t && rank < need) {
            idx[n_gt + rank] = i;
            w[kValAt + n_gt + rank] = tau;
        }
        prefix += total;
        __syncthreads();
    }
}

// Place of each candidate = candidates before it: larger, or equal with a lower
// index.  32 candidates a block (a lane each), the warps share the list.
// DIRECT: the candidates are the values themselves.
template <bool DIRECT>
__global__ void __launch_bounds__(kBlk) rank_kernel(const float* __restrict__ v, int n, const unsigned int* __restrict__ w,
                                                    int k, long long* __restrict__ out_idx, float* __restrict__ out_val) {
    __shared__ unsigned int part[kBlk / 32][32];
    const int m = DIRECT ? n : (overflown(w) ? k : (int)w[kStateAt + 6]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (32 * (int)blockIdx.x >= m) return;
    const unsigned int* vals = DIRECT ? nullptr : w + kValAt;
    const long long* idxs = DIRECT ? nullptr : reinterpret_cast<const long long*>(w + kIdxAt);
    const int me = min(32 * (int)blockIdx.x + lane, m - 1);
    const unsigned int key = DIRECT ? key_bits(v[me]) : vals[me];
    const long long id = DIRECT ? me : idxs[me];
    unsigned int before = 0;
    const int per = ((m + 7) / 8 + 3) & ~3, lo = warp * per, hi = min(m, lo + per);
    auto step = [&](unsigned int x, int j) {
        before += x > key ? 1u : 0u;
        if (x == key) before += (DIRECT ? (long long)j : idxs[j]) < id ? 1u : 0u;
    };
    int j = lo;
    if (!DIRECT) {
#pragma unroll 4
        for (; j + 4 <= hi; j += 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(vals + j);
            step(x.x, j);
            step(x.y, j + 1);
            step(x.z, j + 2);
            step(x.w, j + 3);
        }
    }
#pragma unroll 4
    for (; j < hi; ++j) step(DIRECT ? key_bits(v[j]) : vals[j], j);
    part[warp][lane] = before;
    __syncthreads();
    if (warp == 0 && 32 * (int)blockIdx.x + lane < m) {
        unsigned int r = 0;
        for (int i = 0; i < kBlk / 32; ++i) r += part[i][lane];
        if (r < (unsigned int)k) {
            out_idx[r] = id;
            out_val[r] = __uint_as_float(key);
        }
    }
}

}  // namespace

int topk_launches(long long n, int k) { return k <= 0 || n <= 0 ? 0 : n <= kDirect ? 1 : 9; }

cudaError_t launch_topk(const float* v, long long n, int k, TopkWork& t, cudaStream_t s) {
    if (k <= 0 || n <= 0) return cudaSuccess;
    if (n <= kDirect) {
        rank_kernel<true><<<((int)n + 31) / 32, kBlk, 0, s>>>(v, (int)n, nullptr, k, t.out_idx, t.out_val);
        return cudaGetLastError();
    }
    unsigned int* w = t.scratch;
    cudaError_t e = cudaMemsetAsync(w, 0, sizeof(unsigned int) * kKeyAt, s);
    if (e != cudaSuccess) return e;
    Grouped g{v, n, (int)(((uintptr_t)v & 15u) / 4u), 2, 0};
    while (((g.lead + n - 1) >> g.shift) >= kGroups) ++g.shift;
    g.groups = (int)((g.lead + n - 1) >> g.shift) + 1;
    const int sms = current_sm_count();
    const int bshift = std::max(g.shift, 7) + 4;   // values of a block: 16 warps
    const long long spread = (long long)g.groups << g.shift;
    group_max_kernel<<<(int)(((spread - 1) >> bshift) + 1), 512, 0, s>>>(g, w);
    pivot_kernel<<<1, 1024, 0, s>>>(w, g.groups, (unsigned int)k);
    gather_kernel<<<4 * sms, kBlk, 0, s>>>(g, w);
    const int hgrid = sms * 8;
    hist_kernel<0><<<hgrid, kBlk, 0, s>>>(g, w, (unsigned int)k);
    hist_kernel<1><<<hgrid, kBlk, 0, s>>>(g, w, (unsigned int)k);
    hist_kernel<2><<<hgrid, kBlk, 0, s>>>(g, w, (unsigned int)k);
    const long long per_block = (n + kTieBlocks - 1) / kTieBlocks;
    collect_kernel<<<kTieBlocks, kBlk, 0, s>>>(v, n, per_block, w, (unsigned int)k);
    tie_kernel<<<kTieBlocks, kBlk, 0, s>>>(v, n, per_block, w);
    rank_kernel<false><<<kCand / 32, kBlk, 0, s>>>(v, 0, w, k, t.out_idx, t.out_val);
    return cudaGetLastError();
}


// ---------------------------------------------------------------------------
// Toplist without device allocation: the same launch sequence as above, with
// its scratch in one static device array instead of a context buffer.
namespace {
static_assert(kTopkScratch == 413952, "scratch size stated in fstat_noalloc.h");
static_assert(FSTAT_NOALLOC_MAX_K < kCand, "a list fits the candidate slots");
constexpr int kNaMaxDevices = 64;

std::mutex g_na_mutex;
void* g_na_addr[kNaMaxDevices] = {};
}  // namespace
}  // namespace fs

static __device__ __align__(256) unsigned char g_noalloc_scratch[fs::kTopkScratch];

namespace {
int na_fail(char* msg, int32_t msg_len, int code, const char* text, long long a = 0, long long b = 0) {
    if (msg && msg_len > 0) snprintf(msg, (size_t)msg_len, text, a, b);
    return code;
}
}  // namespace

extern "C" int fstat_toplist_noalloc(int device, const float* v, int64_t n, int32_t k, int64_t* idx_out,
                                     float* val_out, void* cuda_stream, char* msg, int32_t msg_len) {
    using namespace fs;
    if (msg && msg_len > 0) msg[0] = 0;
    if (!v || !idx_out || !val_out) return na_fail(msg, msg_len, FSTAT_EINVAL, "null array pointer");
    if (((uintptr_t)v & 3u) || ((uintptr_t)val_out & 3u) || ((uintptr_t)idx_out & 7u))
        return na_fail(msg, msg_len, FSTAT_EINVAL,
                       "misaligned array: v and val_out need 4-byte, idx_out 8-byte alignment");
    if (k > FSTAT_NOALLOC_MAX_K)
        return na_fail(msg, msg_len, FSTAT_ERANGE, "k = %lld is above the static scratch limit of %lld", k,
                       FSTAT_NOALLOC_MAX_K);
    if (n < 1 || k < 1 || (int64_t)k > n)
        return na_fail(msg, msg_len, FSTAT_EINVAL, "need 1 <= k <= n (k = %lld, n = %lld)", k, (long long)n);
    int count = 0;
    cudaError_t e = cudaGetDeviceCount(&count);
    if (e != cudaSuccess) return na_fail(msg, msg_len, FSTAT_ECUDA, "cudaGetDeviceCount failed (error %lld)", (long long)e);
    if (device < 0 || device >= count || device >= kNaMaxDevices)
        return na_fail(msg, msg_len, FSTAT_EINVAL, "device %lld not available (%lld devices)", device, count);
    e = cudaSetDevice(device);
    if (e != cudaSuccess) return na_fail(msg, msg_len, FSTAT_ECUDA, "cudaSetDevice(%lld) failed (error %lld)", device, (long long)e);
    unsigned char* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_addr[device]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p)
                return na_fail(msg, msg_len, FSTAT_ECUDA, "cudaGetSymbolAddress of the scratch failed on device %lld (error %lld)",
                               device, (long long)e);
            g_na_addr[device] = p;
        }
        base = static_cast<unsigned char*>(g_na_addr[device]);
    }
    TopkWork w{};
    w.scratch = reinterpret_cast<unsigned int*>(base);
    w.out_idx = reinterpret_cast<long long*>(idx_out);
    w.out_val = val_out;
    e = launch_topk(v, (long long)n, (int)k, w, static_cast<cudaStream_t>(cuda_stream));
    if (e != cudaSuccess) return na_fail(msg, msg_len, FSTAT_ECUDA, "toplist launch failed (error %lld)", (long long)e);
    return FSTAT_OK;
}

