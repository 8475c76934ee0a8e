// Dirichlet accumulation with the window sums on the tcgen05 tensor cores
// (D = 8, uniform spindown grid, column step df P T = 1 bin).
//
// For one (sky point, spindown, sub-bin offset) "row" and one SFT the window
// sum of column c is  P_c = sum_k w_k(kappa_c) X[k0 + c + k],  k = -7 .. 8,
//   w_k(kappa) = sin(pi kappa) / (2 (kappa - k)),  kappa_c = kappa_0 + eps c,
// a 16-tap correlation of the SFT's bins with weights that drift slowly along
// the columns.  With the drift written as a quadratic (|eps (c - 32)| < 4e-3,
// remainder < 3e-7) it is a matrix product over bin positions p:
//   P_c = sum_p [A0 + A1 q_p + A2 q_p^2]_p X_p,    q_p = (p - 48) / 64,
// rows (128) x positions (32 .. 64) times positions x columns (64, real and
// imaginary parts interleaved in fours), so one tcgen05.mma per 16 positions
// and operand pair does the 16 taps of 8192 template.SFT pairs.  What is left
// for the FP32 pipes is the twiddle and the Fa, Fb accumulation.
//
// Operands are FP16 pairs: X = Xh + Xl (scaled per SFT by a power of two),
// A0 = A0h + A0l, products hh + hl + lh (2^-22 relative, the FP32 rounding
// level); A1, A2 carry the drift (at most 1e-2 of the sum) and take one FP16
// term each.  Measured against FP64 on random bins: rms error 7.9e-7 of the
// rms bin at the largest Doppler drift, against 1.8e-6 for the sinc polynomial;
// 2F of whole searches 0.7e-6 against 1.7 to 1.9e-6.
//
// X as a matrix of shifted rows (B[c][k] = X[c + k]) is stored once per SFT in
// 128-byte core matrices G[m] = { row i < 4: Re X[4m+i .. 4m+i+7], row 4 + i:
// Im X[4m+i ..] }; core matrix (column block n, position block k) of the
// product is G[n + 2k], so overlapping descriptors (strides 128 and 256 bytes)
// read the whole operand from 32 bytes a position and no row is ever copied.
//
// A block (one per SM, persistent over its run of tiles of 128 rows x 64 columns
// and SFTs, see block_first) is a pipeline of warps joined by mbarriers, over the SFTs:
//   row constants (2 warps, two rows a lane, up to 8 SFTs ahead): khat and phase
//     bases, kappa, the rows whose windows jump (below);
//   copies (1 warp, 3 SFTs ahead): the window of core matrices that covers all
//     rows, one bulk copy;
//   weights (8 warps: thread = row, warpgroup = half of the 16 taps): A0, A1, A2
//     in FP32, their FP16 parts into one of three operand buffers; q X, q^2 X;
//   products (1 warp): 5 tcgen05.mma per 16 positions into one of two
//     accumulators in tensor memory;
//   sums (8 warps: thread = row x 32 columns): window sums from tensor memory,
//     twiddle, Fa and Fb in registers, added up in tensor memory every 64 SFTs,
//     then 2F.
// A row whose window start jumps inside its 64 columns (khat crosses an
// integer: about 64 eps of the (row, SFT)) has the two taps by which the windows
// differ added by the copying warp into a per-block scratch of Fa, Fb.
//
// Bound: instruction issue (61 % of the active cycles, 6810 warp instructions an SFT
// of 8192 pairs: 40 % sums, 40 % weights) with the latency of the stages; tensor pipe
// 23 %, FMA pipes 45 %.  Against the sinc ring: 4000 sky x 1800 f x 10 spindowns x
// 2400 SFTs 203 ms (8.5e11 pairs/s) against 293; 250 x 1733 x 7 x 2302, FP16 bins,
// 217 Hz 9.1 against 15.7 ms; 2048 x 900 x 1 x 1600 4.1 against 6.9; the 1/8-bin
// patch 2048 x 256 2.1 against 3.1.
// What it took, on 4000 sky x 640 f x 600 SFTs (ring 26 ms): one thread issuing
// copies and products beside its weights 55 ms; a warp of its own for them,
// operands in uniform registers 22; code that fits the instruction caches (rolled
// loops, short waits) and 8 weight warps 18.6; three operand buffers and the row
// constants in warps of their own 17.8.  The register shares, the run's length
// read from shared memory and the epilogue of four columns at a time are part of
// it: other shares 207 to 223 ms on the work unit against 204, the length in a
// register 218, eight columns at a time 225 (spills in the sums).
//
// Every wait is bounded; a give-up raises error flag bit 2 and ends the block.
#include <algorithm>

#include "dirichlet.cuh"
#include "mbar.cuh"

namespace fs {
namespace {

constexpr int kThreads = 640;   // warps: 8 weights, 8 sums, 1 products, 1 copies and window jumps, 2 row constants
// registers: the block starts with kLaunchRegs a thread; all but the sum
// warpgroups give some up to them
constexpr int kLaunchRegs = 96, kGenRegs = 48, kSumRegs = 160, kAuxRegs = 64;
static_assert(256 * kGenRegs + 256 * kSumRegs + 128 * kAuxRegs <= kThreads * kLaunchRegs, "register split of one block");
constexpr int kRows = kTcRows, kCols = kTcCols;
constexpr uint32_t kAGroup = kRows * 32;                       // one weight array, 16 positions
constexpr uint32_t kABytes = 36 * kAGroup;                     // weight buffers: three of 3 groups x 4 arrays, or two of 4
constexpr uint32_t kBlk = 256;                                 // core matrices of one 4-position block: high, low part
constexpr uint32_t kXStage = kTcBlkMax * kBlk, kYStage = (kTcBlkMax - 1) * kBlk;
// Fa, Fb go from registers into sums in tensor memory every kFlush SFTs: their
// rounding grows with the root of a register sum's length (2F error against FP64:
// 1.1e-6 without, 0.65e-6 with, 1600 to 2400 SFTs; no change in time).
constexpr int kFlush = 64;
constexpr int kStages = 4, kAhead = 3, kRing = 8;              // SFT stages, SFTs copied ahead, row-constant slots
constexpr uint32_t kOffX = kABytes;
constexpr uint32_t kOffY = kOffX + kStages * kXStage;
constexpr uint32_t kOffP4 = kOffY + 2 * kYStage;               // phase, its column step, twiddle step of 4 columns
constexpr uint32_t kOffW4 = kOffP4 + kRing * kRows * 16;       // kappa at column 32, its column step, first tap's position, a
constexpr uint32_t kOffB = kOffW4 + kRing * kRows * 16;        // b
constexpr uint32_t kOffWin = kOffB + kRing * kRows * 4;
constexpr uint32_t kOffMM = kOffWin + kRing * 8;
constexpr uint32_t kOffEv = kOffMM + kRing * 16;               // rows with a window jump, a bit each
constexpr uint32_t kOffCov = kOffEv + kRing * 16;              // covered templates [x, y)
constexpr uint32_t kOffBar = kOffCov + kRing * 8;
constexpr uint32_t kOffCtrl = kOffBar + 36 * 8;
constexpr uint32_t kSmem = kOffCtrl + 16;
static_assert(kOffX % 128 == 0 && kOffY % 128 == 0 && kOffP4 % 16 == 0 && kOffBar % 8 == 0, "shared-memory layout");
static_assert(kSmem <= 227 * 1024, "shared memory of one block");
// instruction descriptor: D F32, A and B FP16, both K-major, N = 2 kCols, M = 128
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(2 * kCols / 8) << 17) | ((uint32_t)(kRows / 16) << 24);

// Shared-memory descriptors (K-major, no swizzle).  Low word: start address and
// the step to the next 8 positions, in 16-byte units; high word: the step to
// the next 8 rows, and the descriptor version bit.  Only the low word varies.
constexpr uint32_t kDescA = 128 / 16 | 1u << 14, kDescB = kBlk / 16 | 1u << 14;
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t step8) { return (saddr >> 4) | (step8 >> 4) << 16; }
// Issued by one elected lane of a converged warp: the operands are the same in
// all lanes and can stay in uniform registers (from a one-lane branch a product
// took 130 cycles to issue against 66 to run).
__device__ __forceinline__ void mma_issue(uint32_t d, uint32_t a, uint32_t b, uint32_t acc) {
    asm volatile(
        "{\n"
        " .reg .pred p, q;\n"
        " .reg .b64 da, db;\n"
        " mov.b64 da, {%1, %5};\n"
        " mov.b64 db, {%2, %6};\n"
        " setp.ne.u32 p, %4, 0;\n"
        " elect.sync _|q, 0xffffffff;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n"
        "}\n" ::"r"(d),
        "r"(a), "r"(b), "r"(kIdesc), "r"(acc), "n"(kDescA), "n"(kDescB)
        : "memory");
}
// A commit tracks the products of the thread that issues it, so it is issued by
// the lane that the products' election picks (the same for the same mask; which
// one is not specified).
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile(
        "{\n"
        " .reg .pred q;\n"
        " elect.sync _|q, 0xffffffff;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(bar)
        : "memory");
}
// A bounded wait of a few instructions (the kernel has many, in its loops): at
// most 2^21 polls, each held by the hardware for about a microsecond (two to
// three seconds in all).
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p, q;\n"
        " .reg .u32 i;\n"
        " mov.u32 i, 0;\n"
        "POLL_%=:\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " add.u32 i, i, 1;\n"
        " setp.lt.u32 q, i, 2097152;\n"
        " @p bra DONE_%=;\n"
        " @q bra POLL_%=;\n"
        "DONE_%=:\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
          "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
        : "r"(addr));
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"f"(v[0]),
        "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]), "f"(v[10]),
        "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "r"(addr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// the loaded registers pass through the wait, so nothing uses them before it
__device__ __forceinline__ void tmem_wait16(float (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                   "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])
                 :
                 : "memory");
}
__device__ __forceinline__ uint32_t h2_bits(float2 v) {
    const __half2 h = __floats2half2_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float2 h2_float(uint32_t b) { return __half22float2(*reinterpret_cast<const __half2*>(&b)); }
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// sin(pi u) / 2 for |u| <= 0.51 by its Taylor series (relative error < 1e-7).
__device__ __forceinline__ float half_sinpi(float u) {
    const float t = u * u;
    float s = -3.6852155e-3f;                          // -pi^11 / (2 11!)
    s = fmaf(s, t, 4.10729e-2f);                    // pi^9 / (2 9!)
    s = fmaf(s, t, -2.99632265e-1f);                // -pi^7 / (2 7!)
    s = fmaf(s, t, 1.27508202f);                    // pi^5 / (2 5!)
    s = fmaf(s, t, -2.58385639f);                   // -pi^3 / (2 3!)
    s = fmaf(s, t, 1.57079633f);                    // pi / 2
    return s * u;
}

// Element at table position p of a staged SFT (relative to the window), FP32
// sum of its two FP16 parts.  A block's row i holds positions i .. i + 7 after
// its first, so the few past the last block's own four come from its row 3.
__device__ __forceinline__ float2 staged_bin(const unsigned char* X, int p, int last_blk) {
    const int m = min(p >> 2, last_blk), rem = p - 4 * m, i = min(rem, 3);
    const unsigned char* at = X + m * kBlk + i * 16 + (rem - i) * 2;
    auto half = [&](int o) { return __half2float(*reinterpret_cast<const __half*>(at + o)); };
    return make_float2(half(0) + half(128), half(64) + half(64 + 128));
}

// A row whose kappa = kap + eps (c - 32) leaves [0, 1) at column c: that
// column's window starts one bin away from the one the product used.  The tap
// it lacks minus the tap it has too much, times the twiddle, goes to the
// scratch of the row's column.  Only this warp adds to it, in SFT order.
__device__ __forceinline__ void window_jump(const unsigned char* X, int last_blk, int sh, float kap, float eps,
                                            unsigned int ph, unsigned int dphc, float a, float b, int c,
                                            float4* row_scratch) {
    const float y = fmaf((float)(c - 32), eps, kap);
    if (y >= 0.0f && y < 1.0f) return;
    const bool up = y >= 1.0f;
    const float k = up ? y - 1.0f : y + 1.0f;             // kappa in the column's own window
    const float sn = half_sinpi(up ? k : -y);
    const int at = sh + 7 + c + (up ? 1 : -1);            // position of the window's own bin
    const int add = up ? 8 : -7, rem = up ? -8 : 9;
    const float2 xa = staged_bin(X, at + add, last_blk), xr = staged_bin(X, at + rem, last_blk);
    const float wa = sn / (k - (float)add), wr = sn / (k - (float)rem);
    const float pr = wa * xa.x - wr * xr.x, pi = wa * xa.y - wr * xr.y;
    float sp, cp;
    // ph carries the parity of the product's window; this one starts one bin away
    __sincosf((float)(int)(ph + (unsigned int)c * dphc + 0x80000000u) * kPhaseToRad, &sp, &cp);
    const float zr = cp * pr + sp * pi, zi = cp * pi - sp * pr;
    float* f = reinterpret_cast<float*>(row_scratch + c);
    atomicAdd(f, a * zr);
    atomicAdd(f + 1, a * zi);
    atomicAdd(f + 2, b * zr);
    atomicAdd(f + 3, b * zi);
}

// Half of a row's weights: their FP16 parts into the operand buffer.  Positions
// are taken by their residue mod 16 (every row has one tap of each), 0 .. 7 or
// 8 .. 15; arrays of `arr` bytes.
__device__ __forceinline__ void put_weights(unsigned char* A, uint32_t arr, int half, int sh, int gk, float kap, float eps) {
    const int sg = sh >> 4, rho = sh & 15;
    // positions m < rho of a group of 16 belong to the next group
    const int rh = rho - 8 * half;
    const float r0 = (float)(-7 - rho + 8 * half), r1 = r0 + 16.0f;
    const float e0 = eps * (float)(16 - 16 * sg - 8 * half), e1 = fmaf(-16.0f, eps, e0);
    const float sn = half_sinpi(kap <= 0.5f ? kap : 1.0f - kap);
    const float cs = 1.57079633f * __cosf(3.14159265f * kap);
    const float2 s2 = dup(-sn), c2 = dup(-cs), q2 = dup(4.93480220f * sn);
    const float2 E = dup(64.0f * eps), EE = dup(4096.0f * eps * eps);
    const bool next = sg + 1 < gk;
    uint32_t wv[4][4], mk[4];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
        const int m = 2 * jj;
        const bool u0 = m < rh, u1 = m + 1 < rh;
        // k - kappa (k exact)
        const float2 x = make_float2(((u0 ? r1 : r0) + (float)m) - kap, ((u1 ? r1 : r0) + (float)(m + 1)) - kap);
        const float2 rc = make_float2(rcp_approx(x.x), rcp_approx(x.y));
        const float2 w = __fmul2_rn(s2, rc);                   // sin / (2 (kappa - k))
        const float2 w1 = __fmul2_rn(__fadd2_rn(w, c2), rc);   // its derivative
        const float2 w2 = __fmul2_rn(__fadd2_rn(q2, w1), rc);  // half its second derivative
        const float2 ed = make_float2(fmaf((float)-m, eps, u0 ? e1 : e0), fmaf((float)-(m + 1), eps, u1 ? e1 : e0));
        const float2 t = __ffma2_rn(ed, w2, w1);
        const float2 A0 = __ffma2_rn(ed, t, w);
        const float2 A1 = __fmul2_rn(E, __ffma2_rn(ed, w2, t));
        const float2 A2 = __fmul2_rn(EE, w2);
        wv[0][jj] = h2_bits(A0);
        const float2 hb = h2_float(wv[0][jj]);
        wv[1][jj] = h2_bits(make_float2(A0.x - hb.x, A0.y - hb.y));
        wv[2][jj] = h2_bits(A1);
        wv[3][jj] = h2_bits(A2);
        mk[jj] = __funnelshift_lc(0u, 0xffffffffu, 16 * max(rh - m, 0));
    }
#pragma unroll
    for (int ar = 0; ar < 4; ++ar) {
        *reinterpret_cast<uint4*>(A + sg * kAGroup + ar * arr) =
            make_uint4(wv[ar][0] & mk[0], wv[ar][1] & mk[1], wv[ar][2] & mk[2], wv[ar][3] & mk[3]);
        if (next)
            *reinterpret_cast<uint4*>(A + (sg + 1) * kAGroup + ar * arr) =
                make_uint4(wv[ar][0] & ~mk[0], wv[ar][1] & ~mk[1], wv[ar][2] & ~mk[2], wv[ar][3] & ~mk[3]);
    }
#pragma unroll 1
    for (int q = 0; q < gk; ++q) {
        if (q == sg || q == sg + 1) continue;
#pragma unroll
        for (int ar = 0; ar < 4; ++ar)
            *reinterpret_cast<uint4*>(A + ar * arr + q * kAGroup) = make_uint4(0u, 0u, 0u, 0u);
    }
    // the tap next to kappa, where the quotients above cancel: series in x = kappa - k
    const bool one = kap > 0.5f;
    const float x = one ? kap - 1.0f : kap;
    const int kw = sh + (one ? 8 : 7);
    if (fabsf(x) < 0.1f && ((kw >> 3) & 1) == half) {
        const float sg1 = one ? -1.57079633f : 1.57079633f;
        const float xx = x * x;
        const float w = sg1 * fmaf(xx, fmaf(xx, fmaf(xx, -0.190751824f, 0.811742426f), -1.64493407f), 1.0f);
        const float w1 = sg1 * x * fmaf(xx, 3.24696970f, -3.28986813f);
        const float w2 = sg1 * fmaf(xx, 4.87045455f, -1.64493407f);
        const float ed = eps * (float)(16 - kw);
        const float t = fmaf(ed, w2, w1), A0 = fmaf(ed, t, w);
        unsigned char* at = A + (kw >> 4) * kAGroup + (kw & 7) * 2;
        const __half h = __float2half_rn(A0);
        *reinterpret_cast<__half*>(at) = h;
        *reinterpret_cast<__half*>(at + arr) = __float2half_rn(A0 - __half2float(h));
        *reinterpret_cast<__half*>(at + 2 * arr) = __float2half_rn(64.0f * eps * fmaf(ed, w2, t));
        *reinterpret_cast<__half*>(at + 3 * arr) = __float2half_rn(4096.0f * eps * eps * w2);
    }
}

__device__ __forceinline__ void prefetch_l1(const void* q) { asm volatile("prefetch.global.L1 [%0];" ::"l"(q)); }

// The steps (tile x column block, SFT), SFTs fastest, are dealt to the blocks in
// equal runs, so that the last wave of tiles is no emptier than the others (2048 x
// 900 x 1600, 240 tiles on 152 SMs: 5.2 -> 4.6 ms with the search's other kernels).  A
// run starts and ends inside a tile: its first and last segment may hold part of
// the SFTs.  They leave their sums in the scratch, in slot 0 (first segment) and
// slots 1, 2 in turn (the others), for finish_kernel.
constexpr int kScr = kRows * kCols, kSlots = kTcSlots;
__device__ __forceinline__ long long block_first(const TcParams& p, unsigned b, unsigned blocks) {
    return (long long)p.n_tiles * p.n_colb * p.n_sft * b / blocks;
}
// This block's first step, computed where it is used: the sum warps have no
// register to keep it in.
__device__ __forceinline__ long long run_first(const TcParams& p) {
    unsigned b = blockIdx.x;
    asm volatile("" : "+r"(b));
    return block_first(p, b, gridDim.x);
}
__device__ __forceinline__ int seg_slot(int seg) { return seg == 0 ? 0 : 2 - (seg & 1); }

// Where the 2F of a tile's row go: out[j], j < n_live (0: row of padding).
struct RowOut {
    float* out;
    float4 cm;              // combine weights, without coverage
    const float4* cm_j;     // with coverage: by template
    int u, n_live;
};
__device__ __forceinline__ RowOut row_out(const TcParams& p, int item, int row) {
    const int gr = (item % p.n_tiles) * p.rt + row;
    const bool live = row < p.rt && gr < p.n_sky * p.rps;
    const int place = (live ? gr : 0) / p.rps, rr = (live ? gr : 0) - place * p.rps;
    const int d = rr / p.n_sub, sky = p.perm ? p.perm[place] : place;
    return RowOut{p.twoF + ((size_t)sky * p.n_fdot + d) * p.n_f, p.comb[sky], p.comb_j + (size_t)sky * p.n_f, rr - d * p.n_sub,
                  live ? p.n_f : 0};
}
__device__ __forceinline__ float two_f(float4 cm, float4 F) {
    const float f = cm.x * fmaf(F.x, F.x, F.y * F.y) + cm.y * fmaf(F.z, F.z, F.w * F.w) + cm.z * fmaf(F.x, F.z, F.y * F.w);
    return fmaxf(f, 0.0f);
}

// 2F of the tiles whose SFTs were shared by several blocks: block x takes the
// tile that block x of the sums (of `blocks`) began and did not end, adds the
// parts in SFT order, y taking a share of the rows.
__global__ void __launch_bounds__(256) finish_kernel(const TcParams p, int blocks) {
    const int b = blockIdx.x;
    const long long t0 = block_first(p, b, blocks), t1 = block_first(p, b + 1, blocks);
    if (t1 <= t0) return;
    const int item = (int)((t1 - 1) / p.n_sft);
    const long long first = (long long)item * p.n_sft, end = first + p.n_sft;
    if (first < t0 || end <= t1) return;   // begun by another block, or whole
    const int slot = seg_slot(item - (int)(t0 / p.n_sft));
    const int c0 = (item / p.n_tiles) * kCols;
    const int col = threadIdx.x & (kCols - 1);
    for (int row = blockIdx.y * 4 + (threadIdx.x >> 6); row < kRows; row += gridDim.y * 4) {
        const RowOut o = row_out(p, item, row);
        const int j = p.n_sub * (c0 + col) + o.u;
        if (j >= o.n_live) continue;
        float4 F = __ldcg(p.scratch + ((size_t)b * kSlots + slot) * kScr + row * kCols + col);
        for (int q = b + 1; q < blocks && block_first(p, q, blocks) < end; ++q) {
            const float4 x = __ldcg(p.scratch + (size_t)q * kSlots * kScr + row * kCols + col);
            F = make_float4(F.x + x.x, F.y + x.y, F.z + x.z, F.w + x.w);
        }
        o.out[j] = two_f(p.cov ? o.cm_j[j] : o.cm, F);
    }
}

// COV: per-SFT frequency coverage; an SFT's templates j outside [x, y) add nothing.
// A warp whose columns are not all covered sets the others' window sums to zero in
// tensor memory first; the products run on.  1: one template a bin (rows without a
// sub-bin offset, whose lookup in the copying warp cost 4 %), 2: several.  300 sky x
// 1800 f x 5 x 2400, a fifth of the SFTs covering part of the band: 8.7 ms against
// 12.4 ms with the ring that skips; 8.4 without coverage.
template <int COV>
__global__ void __launch_bounds__(kThreads, 1) dirichlet_tc_kernel(const TcParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sb = smem_u32(smem);
    auto bar = [&](unsigned i) { return sb + kOffBar + 8u * i; };
    auto x_full = [&](unsigned n) { return bar(n & 3); };          // [4] SFT copied
    auto r_full = [&](unsigned n) { return bar(4 + (n & 7)); };    // [8] row constants written
    auto r_free = [&](unsigned n) { return bar(12 + (n & 7)); };   // [8] row constants read by the last of their readers
    auto a_full = [&](unsigned n) { return bar(20 + (n & 1)); };   // [2] operands written
    auto a_free = [&](unsigned b) { return bar(22 + b); };         // [3] weights read by the products
    auto d_full = [&](unsigned n) { return bar(25 + (n & 1)); };   // [2] products done
    auto d_free = [&](unsigned n) { return bar(27 + (n & 1)); };   // [2] products read
    auto t_full = [&](int i) { return bar(29 + (i & 1)); };        // [2] tile's window jumps all in place
    auto x_free = [&](unsigned n) { return bar(31 + (n & 3)); };   // [4] SFT's bins read by the products and the window jumps
    const uint32_t fin = bar(35);                                  // last products done
    uint32_t* ctrl = reinterpret_cast<uint32_t*>(smem + kOffCtrl); // [0] tensor-memory address, [1] steps
    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(sb + kOffCtrl) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const long long t0 = block_first(p, blockIdx.x, gridDim.x);
    const unsigned n_steps = (unsigned)(block_first(p, blockIdx.x + 1, gridDim.x) - t0);
    const int item0 = (int)(t0 / p.n_sft), sft0 = (int)(t0 - (long long)item0 * p.n_sft);   // the run's first step
    if (tid == 0) {
        ctrl[1] = n_steps;
        for (int i = 0; i < 4; ++i) {
            mbar_init(x_full(i), 1);
            mbar_init(x_free(i), 2);
        }
        for (int i = 0; i < 8; ++i) {
            mbar_init(r_full(i), 2);
            mbar_init(r_free(i), 9);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(a_full(i), 8);
            mbar_init(d_full(i), 1);
            mbar_init(d_free(i), 8);
            mbar_init(t_full(i), 1);
        }
        for (int i = 0; i < 3; ++i) mbar_init(a_free(i), 1);
        mbar_init(fin, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the block's scratch of window-jump corrections (slot of a segment: seg_slot)
    float4* scratch = p.scratch + (size_t)blockIdx.x * kSlots * kScr;
    const int n_segs = (int)((sft0 + (long long)n_steps - 1) / p.n_sft) + 1;
    for (int i = tid; i < min(n_segs, kSlots) * kScr; i += kThreads) __stcg(scratch + i, make_float4(0.f, 0.f, 0.f, 0.f));
    __threadfence();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = ctrl[0];
    const int row = tid & 127;
    int2* win = reinterpret_cast<int2*>(smem + kOffWin);   // [8] first block, position groups of an SFT
    int2* mm = reinterpret_cast<int2*>(smem + kOffMM);     // [8][2 warps] lowest and highest first position of the rows
    int2* cvr = reinterpret_cast<int2*>(smem + kOffCov);   // [8]
    const float4* P4 = reinterpret_cast<const float4*>(smem + kOffP4);
    const float4* W4 = reinterpret_cast<const float4*>(smem + kOffW4);
    const float* B1 = reinterpret_cast<const float*>(smem + kOffB);
    const uint32_t a_arr = (uint32_t)p.gk * kAGroup;       // a weight buffer holds 4 arrays of gk groups
    const int n_buf = p.gk <= 3 ? 3 : 2;
    // a give-up is uniform over the warp, whose later steps are warp-wide
    auto wait = [&](uint32_t at, unsigned phase) { return __all_sync(0xffffffffu, wait_bar(at, phase & 1u)) != 0; };
    bool ok = true;
    unsigned n = 0;   // steps so far

    if (warp < 8) {
        // ---- weights: thread = row, warpgroup = half of the taps ----------------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kGenRegs));
        int buf = 0;              // weight buffer of SFT n
        unsigned turn = 0;        // its uses so far
        for (; n < ctrl[1]; ++n) {
            ok = wait(r_full(n), n >> 3) && wait(x_full(n), n >> 2) &&      // window known
                 (turn == 0 || wait(a_free(buf), turn - 1));
            if (!ok) break;
            const float4 w = W4[(n & 7) * kRows + row];
            const int2 wn = win[n & 7];
            int sh = __float_as_int(w.z) - 4 * wn.x;
            if (sh < 0 || sh > 16 * wn.y - 16) {   // cannot happen with the planner's bounds
                atomicOr(p.err, 1);
                sh = max(0, min(sh, 16 * wn.y - 16));
            }
            put_weights(smem + buf * 4 * a_arr + (warp >> 2) * (kAGroup / 2) + (row >> 3) * 128 + (row & 7) * 16, a_arr,
                        warp >> 2, sh, wn.y, w.x, w.y);
            if (++buf == n_buf) {
                buf = 0;
                ++turn;
            }
            ok = n < 2 || wait(d_full(n), (n - 2) >> 1);   // the q X buffer is read
            if (!ok) break;
            // q X and q^2 X (first FP16 part only), 16 bytes a thread
            if (tid < (14 + 4 * wn.y) * 8) {
                const uint32_t o = (uint32_t)(tid >> 3) * kBlk + (uint32_t)(tid & 7) * 16;
                const uint4 v = *reinterpret_cast<const uint4*>(smem + kOffX + (n & 3) * kXStage + o);
                const float q0 = (float)(4 * (tid >> 3) + (tid & 3) - 48) * 0.015625f;
                const __half2 q = __floats2half2_rn(q0, q0 + 0.015625f);
                const uint32_t in[4] = {v.x, v.y, v.z, v.w};
                uint32_t y[4], z[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const __half2 qe = __hadd2(q, __floats2half2_rn(0.03125f * e, 0.03125f * e));   // exact
                    const __half2 yy = __hmul2(*reinterpret_cast<const __half2*>(&in[e]), qe);
                    const __half2 zz = __hmul2(yy, qe);
                    y[e] = *reinterpret_cast<const uint32_t*>(&yy);
                    z[e] = *reinterpret_cast<const uint32_t*>(&zz);
                }
                unsigned char* Y = smem + kOffY + (n & 1) * kYStage + o;
                *reinterpret_cast<uint4*>(Y) = make_uint4(y[0], y[1], y[2], y[3]);
                *reinterpret_cast<uint4*>(Y + 128) = make_uint4(z[0], z[1], z[2], z[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(a_full(n));
        }
    } else if (warp >= 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kAuxRegs));
        if (warp == 16) {
            // ---- products ------------------------------------------------------------------------
            int buf = 0;
            for (; n < ctrl[1]; ++n) {
                ok = wait(a_full(n), n >> 1) && (n < 2 || wait(d_free(n), (n - 2) >> 1));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int gk = win[n & 7].y;
                const uint32_t dst = tmem + (n & 1) * (2 * kCols);
                const uint32_t a = desc_lo(sb + buf * 4 * a_arr, kAGroup / 2), arr = a_arr / 16;
                const uint32_t x = desc_lo(sb + kOffX + (n & 3) * kXStage, 2 * kBlk);
                const uint32_t y = desc_lo(sb + kOffY + (n & 1) * kYStage, 2 * kBlk);
                // the accumulator is cut off, not rounded, at each product: the small
                // terms go first, so that few products see its full size (hh first: 2F
                // 5e-7 too small on average).  Offsets in 16-byte units of the start address.
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q < gk) {
                        const uint32_t aq = a + q * (kAGroup / 16), xq = x + q * (4 * kBlk / 16), yq = y + q * (4 * kBlk / 16);
                        mma_issue(dst, aq + 3 * arr, yq + 128 / 16, q);
                        mma_issue(dst, aq + 2 * arr, yq, 1u);
                        mma_issue(dst, aq, xq + 128 / 16, 1u);
                        mma_issue(dst, aq + arr, xq, 1u);
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q < gk) mma_issue(dst, a + q * (kAGroup / 16), x + q * (4 * kBlk / 16), 1u);
                mma_commit(d_full(n));
                mma_commit(a_free(buf));
                mma_commit(x_free(n));
                __syncwarp();
                buf = buf + 1 == n_buf ? 0 : buf + 1;
            }
            mma_commit(fin);
            __syncwarp();
            wait(fin, 0);
        } else if (warp == 17) {
            // ---- copies kAhead SFTs ahead, window jumps ----------------------------------------
            unsigned issued = 0;
            // SFT s of a tile, number q of the block: its window over all rows, and its
            // copy into the stage that the products and the window jumps of SFT q - 4
            // have read.
            auto copy_sft = [&](int s, unsigned q) {
                if (!wait(r_full(q), q >> 3)) return false;
                if (q >= kStages && !wait(x_free(q), (q >> 2) - 1)) return false;
                if (lane == 0) {
                    const int2 u = mm[(q & 7) * 2], v = mm[(q & 7) * 2 + 1];
                    int blk = min(u.x, v.x) >> 2;
                    int gk = (max(u.y, v.y) - 4 * blk + 31) >> 4;
                    if (blk < 0 || gk > p.gk || blk + kTcBlkMax > p.n_blk) {   // cannot happen with the planner's bounds
                        atomicOr(p.err, 1);
                        gk = min(gk, p.gk);
                        blk = max(0, min(blk, p.n_blk - kTcBlkMax));
                    }
                    win[q & 7] = make_int2(blk, gk);
                    if (p.stop < 0 || s < p.stop) {
                        const uint32_t bytes = (uint32_t)(15 + 4 * gk) * kBlk;
                        mbar_expect_tx(x_full(q), bytes);
                        bulk_g2s(sb + kOffX + (q & 3) * kXStage, p.gtab + ((size_t)s * p.n_blk + blk) * kBlk, bytes, x_full(q));
                    }
                }
                __syncwarp();
                if (p.stop < 0 || s < p.stop) issued = q + 1;
                return true;
            };
            int seg = 0, s = sft0, nxt = s;   // SFT of this step, of the next copy
            for (unsigned q = 0; q < kAhead && q < n_steps && ok; ++q) {
                ok = copy_sft(nxt, q);
                nxt = nxt + 1 == p.n_sft ? 0 : nxt + 1;
            }
            for (; n < n_steps && ok; ++n) {
                float4* scr = scratch + seg_slot(seg) * kScr;
                if (n + kAhead < n_steps) ok = copy_sft(nxt, n + kAhead);
                nxt = nxt + 1 == p.n_sft ? 0 : nxt + 1;
                ok = ok && wait(x_full(n), n >> 2);
                if (!ok) break;
                const int2 wn = win[n & 7];
                const unsigned char* X = smem + kOffX + (n & 3) * kXStage;
#pragma unroll 1
                for (int r = 0; r < 4; ++r) {
                    uint32_t ev = *reinterpret_cast<const uint32_t*>(smem + kOffEv + (n & 7) * 16 + 4 * r);
                    while (ev) {   // the lanes take the columns
                        const int src = 32 * r + __ffs(ev) - 1;
                        ev &= ev - 1;
                        const float4 u = W4[(n & 7) * kRows + src], e4 = P4[(n & 7) * kRows + src];
                        const float b = B1[(n & 7) * kRows + src];
                        const int sh = max(0, min(__float_as_int(u.z) - 4 * wn.x, 16 * wn.y - 16));
                        // first column's template of the row, from the tile's first
                        const int jr = COV == 2 ? (((item0 + seg) % p.n_tiles) * p.rt + src) % p.rps % p.n_sub : 0;
#pragma unroll 2
                        for (int c = lane; c < kCols; c += 32) {
                            if (COV && (jr + p.n_sub * c < cvr[n & 7].x || jr + p.n_sub * c >= cvr[n & 7].y)) continue;
                            window_jump(X, 14 + 4 * wn.y, sh, u.x, u.y, __float_as_uint(e4.x), __float_as_uint(e4.y), u.w,
                                        b, c, scr + src * kCols);
                        }
                    }
                }
                const bool last = s + 1 == p.n_sft || n + 1 == n_steps;
                if (last) __threadfence();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(r_free(n));
                    mbar_arrive(x_free(n));
                    if (last) mbar_arrive(t_full(seg));
                }
                seg += last;
                s = s + 1 == p.n_sft ? 0 : s + 1;
            }
            if (!ok) {
                // copies still in flight land before the block retires
                for (unsigned q = issued > 4 ? issued - 4 : 0; q < issued; ++q) wait(x_full(q), q >> 2);
            }
        } else {
            // ---- row constants: two rows a thread, up to kRing SFTs ahead --------------------
            const int rw0 = (warp - 18) * 64 + lane;   // the thread's rows rw0 and rw0 + 32
            int s0 = sft0;
            for (int item = item0; n < n_steps && ok; ++item, s0 = 0) {
                const int s1 = (int)min((unsigned)p.n_sft, s0 + (n_steps - n));
                const int tile = item % p.n_tiles, c0 = (item / p.n_tiles) * kCols;
                auto row_of = [&](int rw, int& place, int& d, int& j0) {
                    const int g = min(tile * p.rt + min(rw, p.rt - 1), p.n_sky * p.rps - 1);
                    place = g / p.rps;
                    const int rr = g - place * p.rps;
                    d = rr / p.n_sub;
                    j0 = rr - d * p.n_sub + p.n_sub * c0;
                };
                int place0, d0, j00, place1, d1, j01;
                row_of(rw0, place0, d0, j00);
                row_of(rw0 + 32, place1, d1, j01);
                for (int s = s0; s < s1; ++s, ++n) {
                    if (n >= kRing) ok = wait(r_free(n), (n - kRing) >> 3);
                    if (!ok) break;
                    const float isc = __ldg(p.inv_scale + s);
                    int lo = 0x7fffffff, hi = -0x7fffffff;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {   // unrolled: both rows' loads fly together
                        const int d = h ? d1 : d0, j0 = h ? j01 : j00;
                        const size_t o = (size_t)s * p.n_sky + (h ? place1 : place0);
                        const longlong2 k = __ldg(reinterpret_cast<const longlong2*>(p.base + o));
                        const uint2 b = __ldg(reinterpret_cast<const uint2*>(&p.base[o].ph0));
                        const long long dk = __ldg(&p.meta[o].dk);
                        const uint4 m = __ldg(reinterpret_cast<const uint4*>(&p.meta[o].dphi));   // dphi, eps, rot
                        const float2 ab = __ldg(reinterpret_cast<const float2*>(&p.meta[o].a));
                        if (s + 2 < p.n_sft) {
                            prefetch_l1(p.base + o + 2 * (size_t)p.n_sky);
                            prefetch_l1(p.meta + o + 2 * (size_t)p.n_sky);
                        }
                        const long long kh = k.x + (long long)d * k.y + (long long)j0 * dk;
                        const int k0 = (int)(kh >> 32);
                        const int pos = k0 - (int)p.k_lo - 7 + p.xoff;
                        lo = min(lo, pos);
                        hi = max(hi, pos);
                        const float eps = 0.25f * __uint_as_float(m.y);
                        const float kap = fmaf(32.0f, eps, (float)(unsigned int)kh * 2.3283064365386963e-10f);
                        const unsigned int ph = b.x + (unsigned int)d * b.y + (unsigned int)j0 * m.x + ((unsigned int)k0 << 31);
                        const unsigned int dphc = (unsigned int)p.n_sub * m.x + 0x80000000u;
                        const int at = (int)(n & 7) * kRows + rw0 + 32 * h;
                        *reinterpret_cast<uint4*>(smem + kOffP4 + at * 16) = make_uint4(ph, dphc, m.z, m.w);
                        *reinterpret_cast<float4*>(smem + kOffW4 + at * 16) =
                            make_float4(kap, eps, __int_as_float(pos), ab.x * isc);
                        *reinterpret_cast<float*>(smem + kOffB + at * 4) = ab.y * isc;
                        // kappa leaves [0, 1) at the first or the last column
                        const float y0 = fmaf(-32.0f, eps, kap), y1 = fmaf(31.0f, eps, kap);
                        const uint32_t ev = __ballot_sync(0xffffffffu, !(y0 >= 0.0f && y0 < 1.0f && y1 >= 0.0f && y1 < 1.0f));
                        if (lane == 0)
                            *reinterpret_cast<uint32_t*>(smem + kOffEv + (n & 7) * 16 + ((warp - 18) * 2 + h) * 4) = ev;
                    }
                    lo = __reduce_min_sync(0xffffffffu, lo);
                    hi = __reduce_max_sync(0xffffffffu, hi);
                    __syncwarp();
                    if (lane == 0) {
                        if (COV) {   // clamped to the band, from the tile's first template; by both warps, the same
                            const int2 c = __ldg(p.cov + s);
                            cvr[n & 7] = make_int2(max(0, min(c.x, p.n_f)) - p.n_sub * c0,
                                                   c.y >= p.n_f ? 1 << 30 : max(0, c.y) - p.n_sub * c0);
                        }
                        mm[(n & 7) * 2 + warp - 18] = make_int2(lo, hi);
                        mbar_arrive(r_full(n));
                    }
                }
            }
        }
    } else {
        // ---- twiddles and sums: thread = row x 32 columns ---------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSumRegs));
        const int h = (warp - 8) >> 2;
        const uint32_t tbase = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 64u * h;
        const uint32_t sums = tbase + 4 * kCols + 64u * h;   // columns 256 + 128 h: the thread's 32 columns of Fa, Fb
        int seg = 0;
        for (; n < ctrl[1] && ok; ++seg) {
            const unsigned end = min(ctrl[1], n + p.n_sft - (unsigned)((run_first(p) + n) % p.n_sft));
            float2 far[16], fai[16], fbr[16], fbi[16];   // column pairs
            auto clear = [&](int i) { far[i] = fai[i] = fbr[i] = fbi[i] = make_float2(0.f, 0.f); };
            // columns 4k .. 4k + 3 added to v
            auto add4 = [&](int k, float (&v)[16]) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = 2 * k + e;
                    v[2 * e] += far[i].x, v[2 * e + 1] += far[i].y;
                    v[4 + 2 * e] += fai[i].x, v[5 + 2 * e] += fai[i].y;
                    v[8 + 2 * e] += fbr[i].x, v[9 + 2 * e] += fbr[i].y;
                    v[12 + 2 * e] += fbi[i].x, v[13 + 2 * e] += fbi[i].y;
                }
            };
            float zero[16] = {};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                clear(2 * k);
                clear(2 * k + 1);
                tmem_st16(sums + 16 * k, zero);
            }
            tmem_wait_st();
            for (; n < end; ++n) {
                ok = wait(r_full(n), n >> 3);
                if (!ok) break;
                const float4 p4 = P4[(n & 7) * kRows + row];
                const float wa = W4[(n & 7) * kRows + row].w, wb = B1[(n & 7) * kRows + row];
                const unsigned int dphc = __float_as_uint(p4.y);
                unsigned int ph = __float_as_uint(p4.x) + 32u * h * dphc;
                float2 tr[2], ti[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    float s0, q0, s1, q1;
                    __sincosf((float)(int)ph * kPhaseToRad, &s0, &q0);
                    ph += dphc;
                    __sincosf((float)(int)ph * kPhaseToRad, &s1, &q1);
                    ph += dphc;
                    tr[i] = make_float2(q0, q1);
                    ti[i] = make_float2(-s0, -s1);
                }
                const float2 rr = dup(p4.z), ri = dup(p4.w), nri = dup(-p4.w), a2 = dup(wa), b2 = dup(wb);
                ok = wait(d_full(n), n >> 1);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t td = tbase + (n & 1) * (2 * kCols);
                bool any = true;   // some column of the warp is covered
                if (COV && (cvr[n & 7].x > 32 * h * p.n_sub || cvr[n & 7].y < (32 * h + 32) * p.n_sub)) {
                    // not all of the warp's columns are covered: zeros into the others' window sums
                    const int2 cv = cvr[n & 7];
                    any = cv.x < (32 * h + 32) * p.n_sub && cv.y > 32 * h * p.n_sub;   // none: the sums stay
                    if (any) {
                        const int item = (int)((run_first(p) + n) / p.n_sft);
                        const int jr = 32 * h * p.n_sub + ((item % p.n_tiles) * p.rt + row) % p.rps % p.n_sub;
#pragma unroll 1
                        for (int ch = 0; ch < 4; ++ch) {
                            float u[16];
                            tmem_ld16(td + 16 * ch, u);
                            tmem_wait16(u);
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                const int j = jr + p.n_sub * (8 * ch + 4 * (e >> 3) + (e & 3));
                                u[e] = j >= cv.x && j < cv.y ? u[e] : 0.0f;
                            }
                            tmem_st16(td + 16 * ch, u);
                        }
                        tmem_wait_st();
                    }
                }
                if (!COV || any) {
                    float v[2][16];
                    tmem_ld16(td, v[0]);
                    tmem_wait16(v[0]);
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {   // eight columns: twice four real parts, four imaginary parts
                        float (&cv)[16] = v[ch & 1];
                        if (ch < 3) tmem_ld16(td + 16 * (ch + 1), v[(ch + 1) & 1]);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int o = 8 * (q >> 1) + 2 * (q & 1), i = 4 * ch + q;
                            const float2 pr = make_float2(cv[o], cv[o + 1]), pi = make_float2(cv[o + 4], cv[o + 5]);
                            float2& wr = tr[q & 1];
                            float2& wi = ti[q & 1];
                            const float2 nwi = make_float2(-wi.x, -wi.y);
                            const float2 zr = __ffma2_rn(wr, pr, __fmul2_rn(nwi, pi));
                            const float2 zi = __ffma2_rn(wr, pi, __fmul2_rn(wi, pr));
                            far[i] = __ffma2_rn(a2, zr, far[i]);
                            fai[i] = __ffma2_rn(a2, zi, fai[i]);
                            fbr[i] = __ffma2_rn(b2, zr, fbr[i]);
                            fbi[i] = __ffma2_rn(b2, zi, fbi[i]);
                            if (i < 14) {   // four columns on
                                const float2 nr = __ffma2_rn(wr, rr, __fmul2_rn(wi, nri));
                                wi = __ffma2_rn(wr, ri, __fmul2_rn(wi, rr));
                                wr = nr;
                            }
                        }
                        if (ch < 3) tmem_wait16(v[(ch + 1) & 1]);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(d_free(n));
                    mbar_arrive(r_free(n));
                }
                if ((n & (kFlush - 1)) == kFlush - 1) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        float u[16];
                        tmem_ld16(sums + 16 * k, u);
                        tmem_wait16(u);
                        add4(k, u);
                        clear(2 * k);
                        clear(2 * k + 1);
                        tmem_st16(sums + 16 * k, u);
                    }
                    tmem_wait_st();
                }
            }
            if (ok) ok = wait(t_full(seg), (unsigned)seg >> 1);
            if (!ok) break;
            // 2F of the row's columns, window-jump corrections added, and the scratch left
            // at zero; of a part of the SFTs, the sums instead of it
            const long long first = run_first(p), t = first + n;
            const int item = (int)((t - 1) / p.n_sft);
            const long long begin = (long long)item * p.n_sft;
            const bool whole = begin >= first && t == begin + p.n_sft;
            const RowOut o = row_out(p, item, row);
            const int j0 = p.n_sub * ((item / p.n_tiles) * kCols + 32 * h) + o.u;
            float4* rs = scratch + seg_slot(seg) * kScr + row * kCols + 32 * h;
#pragma unroll
            for (int q = 0; q < 8; ++q) {   // four columns at a time: their loads fly together
                float4 x[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = __ldcg(rs + 4 * q + e);
                float u[16];
                tmem_ld16(sums + 16 * q, u);
                tmem_wait16(u);
                add4(q, u);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int c = 4 * q + e;
                    const bool hot = x[e].x != 0.f || x[e].y != 0.f || x[e].z != 0.f || x[e].w != 0.f;
                    x[e] = make_float4(x[e].x + u[e], x[e].y + u[4 + e], x[e].z + u[8 + e], x[e].w + u[12 + e]);
                    const int j = j0 + p.n_sub * c;
                    if (whole && j < o.n_live) o.out[j] = two_f(COV ? o.cm_j[j] : o.cm, x[e]);
                    if (whole) x[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (hot || !whole) __stcg(rs + c, x[e]);
                }
            }
            __threadfence();   // the zeros are in place before the scratch's next tile
        }
    }
    if (!ok && lane == 0) atomicOr(p.err, 4);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 16) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// Table of the bins lo .. hi - 1 of one SFT: its scale 2^e (their largest component
// in [2^13, 2^14)) and the core matrices of Xh and Xl.  A bin outside is zero: no
// weight but zero meets it, and at this scale it might be infinite.
template <int FORM>
__global__ void __launch_bounds__(256) tc_tables_kernel(const typename RawT<FORM>::T* __restrict__ bins, long long row, int lo,
                                                        int hi, int n_blk, int xoff, unsigned char* __restrict__ gtab,
                                                        float* __restrict__ inv_scale) {
    using RT = RawT<FORM>;
    __shared__ float red[8];
    const int s = blockIdx.x;
    const typename RT::T* x = bins + (size_t)s * row;
    float mx = 0.f;
    for (int i = lo + threadIdx.x; i < hi; i += 256) {
        const float2 v = RT::f2(x[i]);
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    for (int i = 0; i < 8; ++i) mx = fmaxf(mx, red[i]);
    const int e = mx > 0.f ? max(-114, min(126, 13 - ilogbf(mx))) : 0;
    const float sc = ldexpf(1.0f, e);
    if (threadIdx.x == 0) inv_scale[s] = ldexpf(1.0f, -e);
    unsigned char* dst = gtab + (size_t)s * n_blk * kBlk;
    for (int i = threadIdx.x; i < n_blk * 8; i += 256) {
        const int b0 = 4 * (i >> 3) + (i & 3) - xoff;   // bin of the row's first element
        const bool im = (i & 4) != 0;
        uint32_t h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float2 c = make_float2(0.f, 0.f);
            const int b = b0 + 2 * k;
            if (b >= lo && b < hi) {
                const float2 v = RT::f2(x[b]);
                c.x = (im ? v.y : v.x) * sc;
            }
            if (b + 1 >= lo && b + 1 < hi) {
                const float2 v = RT::f2(x[b + 1]);
                c.y = (im ? v.y : v.x) * sc;
            }
            h[k] = h2_bits(c);
            const float2 hb = h2_float(h[k]);
            l[k] = h2_bits(make_float2(c.x - hb.x, c.y - hb.y));
        }
        unsigned char* o = dst + (size_t)(i >> 3) * kBlk + (i & 7) * 16;
        *reinterpret_cast<uint4*>(o) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(o + 128) = make_uint4(l[0], l[1], l[2], l[3]);
    }
}

// Range of an SFT's bins.  One power of two scales the whole table, and FP16 ends
// at 2^-24, so a bin keeps 2^-25 at worst, 2^-38 of the largest one: beside a strong
// line the weak bins lose bits, which FP32 bins do not, in windows that do not hold
// the line too: Fa, Fb off by 1.5e-6 for a line 10^6 times the noise, 1.8e-4 for
// 10^8 (rms, relative).  Here: the largest component against that of every 16-bin
// window that is not all zeros.  Up to kRangeMax times, which is a line 46 thousand
// times white noise, the loss stays below 0.9e-7, an eighth of the form's error.
// Windows that hang over the band's edge count with the bins they have; fewer than
// eight (neither bin next to kappa is among them) are often weak by chance, and may be
// kRangeEdge times weaker (loss 1e-5).
// Bound: one read of the bins, only when new bins meet a bank that suits the form.
constexpr float kRangeMax = 65536.0f, kRangeEdge = 64.0f;
constexpr int kRangeRun = 2048;   // windows of a pass, eight a thread
template <int FORM>
__global__ void __launch_bounds__(256) tc_range_kernel(const typename RawT<FORM>::T* __restrict__ bins, long long row,
                                                       int n_bins, int lo, int hi, int* __restrict__ flag) {
    using RT = RawT<FORM>;
    auto at = [](int i) { return i + (i >> 3); };   // threads 9 words apart: no bank conflicts
    __shared__ float mag[kRangeRun + 16 + (kRangeRun + 16) / 8];
    __shared__ float red[2][8];
    const typename RT::T* x = bins + (size_t)blockIdx.x * row;
    float largest = 0.f, quiet = __int_as_float(0x7f800000);
    for (int s0 = lo; s0 == lo || s0 + 15 < hi; s0 += kRangeRun) {   // windows s0 .. , the first one even of a shorter range
        __syncthreads();
        for (int i = threadIdx.x; i < kRangeRun + 15; i += 256) {
            const int b = s0 + i;
            float m = 0.f;
            if (b >= 0 && b < min(n_bins, hi)) {
                const float2 v = RT::f2(x[b]);
                m = fmaxf(fabsf(v.x), fabsf(v.y));
            }
            mag[at(i)] = m;
            largest = fmaxf(largest, m);
        }
        __syncthreads();
        // a thread's windows start at i0 .. i0 + 7: bins 7 .. 15 after i0 are in all of them
        const int i0 = 8 * (int)threadIdx.x;
        float head[8], all = 0.f;
        head[7] = 0.f;
#pragma unroll
        for (int k = 6; k >= 0; --k) head[k] = fmaxf(head[k + 1], mag[at(i0 + k)]);
#pragma unroll
        for (int k = 7; k < 16; ++k) all = fmaxf(all, mag[at(i0 + k)]);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k > 0) all = fmaxf(all, mag[at(i0 + 15 + k)]);
            const float w = fmaxf(all, head[k]);
            const int s = s0 + i0 + k;
            if (w > 0.f && (s + 16 <= hi || s == lo))
                quiet = fminf(quiet, min(s + 16, n_bins) - max(s, 0) < 8 ? kRangeEdge * w : w);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        largest = fmaxf(largest, __shfl_xor_sync(0xffffffffu, largest, o));
        quiet = fminf(quiet, __shfl_xor_sync(0xffffffffu, quiet, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = largest;
        red[1][threadIdx.x >> 5] = quiet;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) {
            largest = fmaxf(largest, red[0][i]);
            quiet = fminf(quiet, red[1][i]);
        }
        if (largest > kRangeMax * quiet) atomicOr(flag, 1);
    }
}

}  // namespace

cudaError_t launch_tc_tables(const void* bins, int form, long long row, int n_sft, int lo, int hi, int n_blk, int xoff,
                             unsigned char* gtab, float* inv_scale, cudaStream_t s) {
    if (form == FSTAT_BINS_C64)
        tc_tables_kernel<FSTAT_BINS_C64><<<n_sft, 256, 0, s>>>(static_cast<const float2*>(bins), row, lo, hi, n_blk, xoff, gtab,
                                                               inv_scale);
    else if (form == FSTAT_BINS_F16)
        tc_tables_kernel<FSTAT_BINS_F16><<<n_sft, 256, 0, s>>>(static_cast<const __half2*>(bins), row, lo, hi, n_blk, xoff, gtab,
                                                               inv_scale);
    else
        tc_tables_kernel<FSTAT_BINS_BF16><<<n_sft, 256, 0, s>>>(static_cast<const __nv_bfloat162*>(bins), row, lo, hi, n_blk,
                                                                xoff, gtab, inv_scale);
    return cudaGetLastError();
}

cudaError_t launch_tc_range(const void* bins, int form, long long row, int n_sft, int n_bins, int lo, int hi, int* flag,
                            cudaStream_t s) {
    if (form == FSTAT_BINS_C64)
        tc_range_kernel<FSTAT_BINS_C64><<<n_sft, 256, 0, s>>>(static_cast<const float2*>(bins), row, n_bins, lo, hi, flag);
    else if (form == FSTAT_BINS_F16)
        tc_range_kernel<FSTAT_BINS_F16><<<n_sft, 256, 0, s>>>(static_cast<const __half2*>(bins), row, n_bins, lo, hi, flag);
    else
        tc_range_kernel<FSTAT_BINS_BF16><<<n_sft, 256, 0, s>>>(static_cast<const __nv_bfloat162*>(bins), row, n_bins, lo, hi,
                                                               flag);
    return cudaGetLastError();
}

// One block an SM, but at least 32 steps a block where there are fewer tiles.
int tc_blocks(int n_tiles, int n_colb, int n_sft, int sms) {
    const long long items = (long long)n_tiles * n_colb;
    return (int)std::min<long long>(sms, std::max(std::min<long long>(items, sms), items * n_sft / 32));
}

int tc_launches(const TcParams& p) {
    const int grid = tc_blocks(p.n_tiles, p.n_colb, p.n_sft, current_sm_count());
    return (long long)p.n_tiles * p.n_colb % grid == 0 ? 1 : 2;   // whole tiles only, or finish_kernel too
}

cudaError_t launch_dirichlet_tc(const TcParams& p, cudaStream_t s) {
    const auto kernel = !p.cov ? dirichlet_tc_kernel<0> : p.n_sub == 1 ? dirichlet_tc_kernel<1> : dirichlet_tc_kernel<2>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    const int grid = tc_blocks(p.n_tiles, p.n_colb, p.n_sft, current_sm_count());
    kernel<<<grid, kThreads, kSmem, s>>>(p);
    if ((e = cudaGetLastError()) != cudaSuccess || tc_launches(p) == 1) return e;
    finish_kernel<<<dim3(grid, 16), 256, 0, s>>>(p, grid);
    return cudaGetLastError();
}

}  // namespace fs
