// The FP64 path's update of a whole batch on the tcgen05 tensor cores, to FP64
// accuracy.
//
// GB300's FP64 pipe issues two lanes per clock and SM: the twelve fused
// multiply-adds of an element-update bound a plain FP64 kernel at 5e10
// updates/s, whatever the memory system does.  The tensor cores reach FP64
// precision through integer arithmetic instead: every operand becomes eight
// signed base-256 digits of a 62-bit integer scaled by one power of two per
// operand row, each digit an FP16 value in [-128, 127] (exact), and the digit
// products are summed in FP32 accumulators that never leave the integers below
// 2^24 -- so every sum is exact.  (The error-free splitting of a matrix product
// into slices with exact partial products is the method of Ozaki, Ogita, Oishi
// and Rump, Numerical Algorithms 59, 2012.)
//
//   x = 2^(e-62) v,  |v| < 2^62,  v = sum_t d_t 256^(7-t),  t = 0..7
//   u w = 2^(eu+ew-124) sum_p 256^(14-p) sum_{s+t=p} d_s(u) d_t(w)
//
// Levels p = 0..7 (36 digit products) are kept, each in its own accumulator.
// With at most 256 terms of K (64 measurements x 2 spins x 2 components) levels
// 0..4 stay below 2^24 whatever the digits are (the leading digit is at most
// 64); levels 5 to 7, whose unit is 2^-52 of the largest product and less,
// could pass 2^24 only if nearly all of 1500 digit products were largest and of
// one sign, and would then round to even integers.  The epilogue puts the eight
// integers together in 96-bit integer arithmetic and rounds once to FP64.
//
// Accuracy.  An operand is exact down to 2^-62 of its row's unit 2^e (the row:
// one G entry over the batch's measurements and spins, real and imaginary part;
// |x| < 2^e), and the dropped levels are below 2^-59 of 2^(eu+ew), 2^-62 in the
// mean: an entry's error is relative to the rows' largest values, where FP64's
// is relative to the products that are summed.  A pass over the staged G before
// the first operand is formed (k_spread) keeps the two together: a batch with a
// row of which more than a quarter of one spin's values lie more than 2^7 below
// the row's largest is left to the plain kernels, as is one with a non-finite G
// entry or a component outside 2^+-380 (one device flag for all of them).  What
// remains has, for half of an entry's products or more, both factors above 2^-8
// of their rows' units, which bounds the error by 2^-40 of the sum of the
// products' moduli, all errors of one sign and all products as small as the
// rule allows.  In the mean, of 128 products, relative to that sum: 4e-19 for
// values of like size (a plain FP64 sum: 4e-17), 1e-16 for one value in each
// row 2^6 above the others, in different measurements (plain: 2e-16).  Seven
// digits and levels without such a check had 1e-16 and 4e-14, and no bound.
//
// The GEMMs are those of the mixed path (g4_exchange_tc.cu, g4_direct_tc.cu):
//   exchange  rows K1 of diagonal D x columns P of diagonal -D, K = (r, spin)
//   direct    rows K1 x columns K2 of one transfer Q, K = r, into an FP64
//             scratch of a few transfers that k_merge64 adds to the accumulator
// with Re and Im interleaved in the rows alone: every operand row is stored as
// (-Im, Re, Im), and the K axis runs over Re w against (Re u, Im u), then Im w
// against (-Im u, Re u), so that an accumulator entry is a finished component
// (interleaved columns as well left two accumulator entries, two conversions
// and a lane exchange per component to an epilogue that bounded the kernel:
// 10.6 ms a batch on the 4x4 cluster with 64 frequencies and 8 transfers).
//
// k_gemm_digits, one CTA per SM, warp roles:
//   warp 0      TMA producer: per 32 values of K one stage of 8 + 8 boxes
//   warp 1      MMA issuer: per stage 36 products x 2 steps of 16 values of K,
//               level by level; eight accumulators of up to 64 columns
//   warps 2..17 epilogue: four per tensor-memory lane quarter, each a quarter
//               of the columns.  A level is drained into integer registers as
//               soon as it is complete and handed back, while the next levels
//               are still being multiplied.
// What bounds it: the MMAs, whose 128-row A operand is read from shared memory
// every time (128 x 64 x 16 per MMA: about 48 clocks of shared-memory reads for
// 32 of arithmetic); eight accumulators of 64 columns fill tensor memory, so N
// cannot be larger; with few values of K the epilogue.  Measured, one batch of
// 64 on the 4x4 cluster with 64 frequencies, 8 x 16 transfers: per-measurement
// launches of the plain tiled kernel 279 ms; here 16.6 ms (exchange 8.8, direct 2.8, packs and spread 3.4,
// merge 1.6).  By ncu (32 frequencies) the tensor pipe is active in 65 to 71% of
// the exchange's cycles.
// Every wait is bounded as in the mixed path's kernels.
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <new>
#include <vector>

#include "g4_diag.cuh"
#include "g4_internal.h"
#include "g4_ptx.cuh"

namespace {

using namespace g4ptx;

constexpr int kDig = 8;                        // base-256 digits of an operand
constexpr int kChunk = 32;                     // K values per stage (64-byte rows)
constexpr int kStages = 2;
constexpr int kARows = 128;
constexpr int kAPlane = kARows * 64;           // bytes of one A digit plane per stage
constexpr int kMaxN = 64;                      // columns per level accumulator
constexpr int kEpiWarps = 16;
constexpr int kThreads = 32 * (2 + kEpiWarps);
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxChunks = 8;
constexpr int kMaxWex = 16;                    // largest Nwex of this path
constexpr int kMinSmem = 116 * 1024;           // two blocks never share an SM (tensor memory)
constexpr int kMaxSmem = 227 * 1024;
constexpr int kSpread = 7;                     // bits of spread within a row, see k_spread

struct FSigns {
    double rs[64];          // sqrt(|s|)
    unsigned char neg[64];  // s < 0: the factor is i sqrt(|s|)
};

// ------------------------------------------------------------------ digits
// |x| < 2^e as v = round(x 2^(62-e)) on the integer pipes.
__device__ __forceinline__ long long to_fixed(double x, int e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7FFu);
    if (eb == 0) return 0;
    const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = eb - 1013 - e;   // v = mant 2^sh, sh <= 9
    unsigned long long v;
    if (sh >= 0) v = mant << sh;
    else if (sh <= -55) v = 0;
    else v = (mant + (1ull << (-sh - 1))) >> -sh;
    return (long long)b < 0 ? -(long long)v : (long long)v;
}

// Digits of the rows of one position: xs = [Re | Im][J] values in shared
// memory, J a multiple of 16; one warp.  Digit t goes to out + t * plane +
// c * J + jj (FP16) for c = 0 (-Im), 1 (Re), 2 (Im); the common exponent to *ex.
// Only the jj below `live` of each half (spin) of J/nhalf values are written.
__device__ __forceinline__ void write_digits(const double* xs, int ld, int J, int nhalf, int live,
                                             __half* out, size_t plane, int* ex) {
    const int lane = threadIdx.x & 31;
    unsigned top = 0;
    for (int i = lane; i < 2 * J; i += 32) {
        const int c = i >= J ? 1 : 0;
        top = max(top, (unsigned)__double2hiint(xs[c * ld + i - c * J]) & 0x7FFFFFFFu);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    const int eb = (int)(top >> 20);
    const int e = eb ? eb - 1022 : 0;
    if (lane == 0) *ex = e;
    const int jq = J / 4, hq = jq / nhalf, lq = live / 4;
    for (int i = lane; i < 2 * jq; i += 32) {
        const int c = i >= jq ? 1 : 0, j = i - c * jq;
        if (j % hq >= lq) continue;
        const double2 a = *reinterpret_cast<const double2*>(xs + c * ld + 4 * j);
        const double2 b = *reinterpret_cast<const double2*>(xs + c * ld + 4 * j + 2);
        const double x[4] = {a.x, a.y, b.x, b.y};
        uint32_t lo[4], hi[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned long long w =
                (unsigned long long)to_fixed(x[u], e) + 0x8080808080808080ull;
            lo[u] = (uint32_t)w;
            hi[u] = (uint32_t)(w >> 32);
        }
        __half* o = out + (size_t)(1 + c) * J + 4 * j;
#pragma unroll
        for (int t = 0; t < kDig; ++t) {
            // byte 7-t of two values into the low bytes of two halves: 1024 + b
            const int by = kDig - 1 - t, n = by & 3;
            const uint32_t sel = (uint32_t)(n | (n << 4) | ((4 + n) << 8) | ((4 + n) << 12));
            const uint32_t p01 = (__byte_perm(by < 4 ? lo[0] : hi[0], by < 4 ? lo[1] : hi[1], sel) & 0x00FF00FFu) | 0x64006400u;
            const uint32_t p23 = (__byte_perm(by < 4 ? lo[2] : hi[2], by < 4 ? lo[3] : hi[3], sel) & 0x00FF00FFu) | 0x64006400u;
            const __half2 bias = __half2half2(__ushort_as_half((unsigned short)0x6480));   // 1152
            uint2 q;
            __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&p01), bias);
            q.x = *reinterpret_cast<uint32_t*>(&h);
            h = __hsub2(*reinterpret_cast<const __half2*>(&p23), bias);
            q.y = *reinterpret_cast<uint32_t*>(&h);
            *reinterpret_cast<uint2*>(o + t * plane) = q;
            if (c) *reinterpret_cast<uint2*>(o + t * plane - 2 * J) = make_uint2(q.x ^ 0x80008000u, q.y ^ 0x80008000u);
        }
    }
}

// Sets *flag when the digits would lose more than FP64 does (see the top of the
// file): a G entry (i, j) -- a row of the exchange operands, and where it is
// one of the direct operands (|n_i - n_j| a transfer of the handle) the spins'
// combination -- of which more than a quarter of the values of one spin lie
// more than 2^kSpread below the row's largest.  Zeros count as small, a row of
// zeros alone does not.  One thread per entry; the exponents of its values are
// kept in shared memory between the search for the largest and the count.
// One read of the staged G: 3.9 TB/s (4x4 cluster, 32 frequencies, 64
// measurements: 0.14 ms).
struct SpreadArgs {
    signed char se[64];   // exponent of a measurement's sign factor; -128: weight zero
};

__global__ void __launch_bounds__(256) k_spread(const double2* __restrict__ G, int staged,
                                                const __grid_constant__ SpreadArgs A, bool direct, G4Dims d,
                                                unsigned* __restrict__ flag) {
    if (*flag) return;
    extern __shared__ unsigned short exps[];   // [3 staged][256]: spin up, spin down, combination
    const size_t NN = (size_t)d.N * d.N;
    const double ws = d.ch == G4_PH_DENSITY ? 1.0 : -1.0;
    unsigned short* ex = exps + threadIdx.x;
    bool bad = false;
    for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < NN; e += (size_t)gridDim.x * 256) {
        const int i = (int)(e / d.N), j = (int)(e - (size_t)i * d.N);
        const int dn = abs(i % d.Nw2 - j % d.Nw2);
        const bool both = direct && dn >= d.m0 && dn < d.m0 + d.Nwex;
        int top = 0, topd = 0;
        auto put = [&](int row, double2 v, int se) {
            const unsigned h = max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu,
                                   (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu) >> 20;
            const int x = h && se > -128 ? max((int)h + se, 1) : 0;
            ex[row * 256] = (unsigned short)x;
            return x;
        };
#pragma unroll 4
        for (int r = 0; r < staged; ++r) {
            const double2 a = G[(size_t)(2 * r) * NN + e], b = G[(size_t)(2 * r + 1) * NN + e];
            const int se = A.se[r];
            top = max(top, max(put(2 * r, a, se), put(2 * r + 1, b, se)));
            if (both) topd = max(topd, put(2 * staged + r, make_double2(a.x + ws * b.x, a.y + ws * b.y), se));
        }
        int c0 = 0, c1 = 0, cd = 0;
        for (int r = 0; r < staged; ++r) {
            c0 += (int)ex[2 * r * 256] < top - kSpread;
            c1 += (int)ex[(2 * r + 1) * 256] < top - kSpread;
            if (both) cd += (int)ex[(2 * staged + r) * 256] < topd - kSpread;
        }
        if (top > 0 && max(c0, c1) > staged / 4) bad = true;
        if (topd > 0 && cd > staged / 4) bad = true;
    }
    if (bad) *flag = 1u;
}

// Exchange operands of one group of diagonals [a0, a0 + na): every G entry
// (i, j) as a row of J = 2 Jh values jj = spin * Jh + r per component, digit
// planes X[(a * 8 + t)][k][n][c][jj], c = (-Im, Re, Im) (a: the group's position of the diagonal
// (kr (-) k, ni - n) for i = (kr, ni), j = (k, n)) and exponents ex[a][k][n].
// A block takes one row i and eight consecutive columns j of one momentum: it
// reads one 128-byte line of every slot and spin, and writes whole rows of X
// (2 J bytes per digit and component).  Values r >= staged are zero, written
// up to the next multiple of 32 (the GEMM's chunks of K).  The group's diagonals
// have dn0 <= |dn| <= dn1, so that a row meets them in two bands of columns:
// blockIdx.x / Nc counts band 0's nband blocks, then band 1's (a launch over all
// columns, left at once by the blocks without one of the group, took 0.28 ms a
// group on the 4x4 cluster with 64 frequencies).  HBM-bound: 16 B
// read and 48 B written per entry, slot and spin.
constexpr int kPackJ = 8;

__global__ void __launch_bounds__(256) k_pack_digits(const double2* __restrict__ G, int staged, int Jh,
                                                     int live, FSigns sg, const int* __restrict__ pos0,
                                                     int a0, int na, int dn0, int dn1, int nband,
                                                     __half* __restrict__ X,
                                                     int* __restrict__ ex, G4Dims d,
                                                     const unsigned* __restrict__ flag) {
    if (*flag) return;
    extern __shared__ __align__(16) double xs[];   // [kPackJ][2][ld]
    const int J = 2 * Jh, ld = J + 2;
    const int i = blockIdx.y, kr = i / d.Nw2, ni = i - kr * d.Nw2;
    const int bx = blockIdx.x / d.Nc, k = blockIdx.x - bx * d.Nc;
    // column blocks of n = ni - dn1 .. ni - dn0, then those of ni + dn0 .. ni + dn1
    // that the first band does not have
    const int end0 = ni - dn0 >= 0 ? (ni - dn0) / kPackJ + 1 : 0;
    int jb;
    if (bx < nband) {
        jb = max(0, ni - dn1) / kPackJ + bx;
        if (jb >= end0) return;
    } else {
        jb = max((ni + dn0) / kPackJ, end0) + bx - nband;
        if (jb * kPackJ > min(d.Nw2 - 1, ni + dn1)) return;
    }
    const int n0 = jb * kPackJ, nv = min(kPackJ, d.Nw2 - n0);
    int dkx = kr % d.Lx - k % d.Lx, dky = kr / d.Lx - k / d.Lx;
    dkx += dkx < 0 ? d.Lx : 0;
    dky += dky < 0 ? d.Ly : 0;
    const int dk = dkx + d.Lx * dky;
    const int mk = (dkx ? d.Lx - dkx : 0) + d.Lx * (dky ? d.Ly - dky : 0);
    bool any = false;   // no column of this block lies in the group
    for (int c = 0; c < nv; ++c) {
        const int a = diag_pos(dk, ni - n0 - c, mk, d.Nc, pos0) - a0;
        any = any || (a >= 0 && a < na);
    }
    if (!any) return;
    const size_t NN = (size_t)d.N * d.N;
    const double2* src = G + (size_t)i * d.N + k * d.Nw2 + n0;
    for (int t = threadIdx.x; t < J * kPackJ; t += blockDim.x) {
        const int c = t & (kPackJ - 1), jj = t / kPackJ;
        const int sp = jj >= Jh ? 1 : 0, r = jj - sp * Jh;
        double2 v = make_double2(0.0, 0.0);
        if (r < staged && c < nv) {
            v = src[(size_t)(2 * r + sp) * NN + c];
            const double f = sg.rs[r];
            if (f != 1.0) {
                v.x *= f;
                v.y *= f;
            }
            if (sg.neg[r]) v = make_double2(-v.y, v.x);
        }
        xs[(c * 2 + 0) * ld + jj] = v.x;
        xs[(c * 2 + 1) * ld + jj] = v.y;
    }
    __syncthreads();
    const int c = threadIdx.x >> 5;
    if (c >= nv) return;
    const int n = n0 + c;
    const int a = diag_pos(dk, ni - n, mk, d.Nc, pos0) - a0;
    if (a < 0 || a >= na) return;
    const size_t row = (size_t)k * d.Nw2 + n;
    const size_t plane = (size_t)d.N * 3 * J;
    write_digits(xs + c * 2 * ld, ld, J, 2, live, X + (size_t)a * kDig * plane + row * 3 * J, plane,
                 ex + (size_t)a * d.N + row);
}

// Direct operands of the transfers Q0 .. Q0 + gridDim.y: a_r(K) (side 0) and
// b_r(K) (side 1) as digit planes P[side][(Ql * 8 + t)][K][c][r], r < Bp, c as above, and
// exponents ex[side][Ql][K].  One block per eight frequencies of one momentum.
__global__ void __launch_bounds__(256) k_pack_digits_ab(const double2* __restrict__ G, int staged, int Bp,
                                                        int live, FSigns sg, int Q0, int nQg,
                                                        __half* __restrict__ P, int* __restrict__ ex,
                                                        G4Dims d, const unsigned* __restrict__ flag) {
    if (*flag) return;
    extern __shared__ __align__(16) double xs[];   // [kPackJ][2][ld]
    const int ld = Bp + 2;
    const int njb = (d.Nw2 + kPackJ - 1) / kPackJ;
    const int k = blockIdx.x / njb, n0 = (blockIdx.x - k * njb) * kPackJ;
    const int Ql = blockIdx.y, Q = Q0 + Ql, side = blockIdx.z;
    const int q = Q / d.Nwex, m = d.m0 + Q - q * d.Nwex;
    const int nv = min(kPackJ, d.Nw2 - n0);
    int kx = k % d.Lx + q % d.Lx, ky = k / d.Lx + q / d.Lx;
    kx -= kx >= d.Lx ? d.Lx : 0;
    ky -= ky >= d.Ly ? d.Ly : 0;
    const int kq = kx + d.Lx * ky;
    const double ws = d.ch == G4_PH_DENSITY ? 1.0 : -1.0;   // weight of spin -1
    const size_t NN = (size_t)d.N * d.N;
    for (int t = threadIdx.x; t < Bp * kPackJ; t += blockDim.x) {
        const int c = t & (kPackJ - 1), r = t / kPackJ, n = n0 + c;
        double2 v = make_double2(0.0, 0.0);
        if (r < staged && c < nv && n + m < d.Nw2) {
            // a: G(K + Q, K); b: G(K, K + Q)
            const size_t e = side ? (size_t)(k * d.Nw2 + n) * d.N + kq * d.Nw2 + n + m
                                  : (size_t)(kq * d.Nw2 + n + m) * d.N + k * d.Nw2 + n;
            const double2 g0 = G[(size_t)(2 * r) * NN + e], g1 = G[(size_t)(2 * r + 1) * NN + e];
            const double f = sg.rs[r];
            v = make_double2(f * (g0.x + ws * g1.x), f * (g0.y + ws * g1.y));
            if (sg.neg[r]) v = make_double2(-v.y, v.x);
        }
        xs[(c * 2 + 0) * ld + r] = v.x;
        xs[(c * 2 + 1) * ld + r] = v.y;
    }
    __syncthreads();
    const int c = threadIdx.x >> 5;
    if (c >= nv) return;
    const size_t row = (size_t)k * d.Nw2 + n0 + c;
    const size_t plane = (size_t)d.N * 3 * Bp;
    write_digits(xs + c * 2 * ld, ld, Bp, 1, live,
                 P + ((size_t)side * nQg + Ql) * kDig * plane + row * 3 * Bp, plane,
                 ex + ((size_t)side * nQg + Ql) * d.N + row);
}

// ------------------------------------------------------------------ GEMM
struct FParams {
    double2* acc;            // exchange: acc[K1][K2][q][m]
    double2* scr;            // direct: [Ql][K1][K2]
    unsigned* status;
    const unsigned* flag;
    const int4* work;        // exchange: per (D, row block) {aD | bD << 16, dk, dn, n0}
    const int* exA;          // exchange: ex[a][k][n]; direct: ex[0][Ql][K]
    const int* exB;          // direct: ex[1][Ql][K]
    int Lx, Ly, Nc, Nw2, N, Nwex, Nkex, NQ, m0;
    int kb, nb, W, pb, nkb, npb;
    int ncols;               // MMA N
    // chunks of K: offset in A and in B, and the component: 0 (Re w), 1 (Im w)
    int nchunk, jA[kMaxChunks], jB[kMaxChunks], cw[kMaxChunks];
    int ntiles, run;
    int bplane;
    uint32_t txbytes, idesc;
    long long budget;
};

// 8 consecutive 32-bit columns of this thread's lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row atoms of
// 512 bytes.
__device__ __forceinline__ uint64_t sdesc_k64(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;                 // SWIZZLE_64B
    return d;
}

__device__ __forceinline__ void bulk_add_f64(double2* gdst, const double2* ssrc, uint32_t bytes) {
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f64 [%0], [%1], %2;" ::"l"(gdst),
                 "r"(smem_u32(ssrc)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Barrier of the four warps of one lane quarter; true if any thread passes
// true (the same answer for all of them).
__device__ __forceinline__ bool quarter_any(int quad, bool p) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %2, 0;\n"
        " barrier.cta.red.or.pred q, %1, 128, p;\n selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"(quad + 1), "r"(p ? 1u : 0u)
        : "memory");
    return r != 0;
}

// (hi, mid, lo) += w 2^(56-8p), level p's part of a 96-bit integer.  Shifts and
// carries: 64-bit multiply-adds took the direct GEMM of one batch on the 4x4
// cluster with 64 frequencies from 2.8 to 3.3 ms.
template <int P>
__device__ __forceinline__ void add_level(uint32_t& lo, uint32_t& mid, uint32_t& hi, int w) {
    constexpr int S = 24 - 8 * (P & 3);
    const uint32_t a = (uint32_t)w << S, b = (uint32_t)(w >> (S ? 32 - S : 31));
    if constexpr (P < 4)
        asm("add.cc.u32 %0, %0, %2;\n addc.u32 %1, %1, %3;" : "+r"(mid), "+r"(hi) : "r"(a), "r"(b));
    else
        asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %4;\n addc.u32 %2, %2, %5;"
            : "+r"(lo), "+r"(mid), "+r"(hi)
            : "r"(a), "r"(b), "r"((uint32_t)(w >> 31)));
}

// (hi, mid, lo) 2^sc in FP64, rounded to nearest (|sc| small enough for a
// normal result), negated when neg is set: the 64 leading bits (|t| < 2^78) go
// through one conversion on the FP64 pipe; what is cut off is below 2^-61 of
// the value.  Scale and sign on the integer pipes (the conversion there as
// well, about 45 instructions, made the epilogue the limit of small batches).
__device__ __forceinline__ double fixed_to_f64(uint32_t lo, uint32_t mid, uint32_t hi, int sc, bool neg) {
    const long long h = (long long)(((unsigned long long)hi << 32) | mid);
    const int s = min(32, __clzll(h ^ (h >> 63)) - 1);   // 17 .. 32
    const long long v = (long long)(((unsigned long long)h << s) | (lo >> (32 - s)));
    const double x = __ll2double_rn(v);
    const int xh = (__double2hiint(x) + (sc + 32 - s) * (1 << 20)) ^ (neg ? (int)0x80000000u : 0);
    return v == 0 ? 0.0 : __hiloint2double(xh, __double2loint(x));
}

struct FTile {
    int aD, bD, dk, dn, n0, kblk, pblk;   // exchange
    int Ql, i0, j0;                       // direct
};

// MODE 0: exchange, particle-hole geometry; 1: exchange, particle-particle; 2: direct.
template <int MODE>
__device__ __forceinline__ FTile f_tile(const FParams& P, int t) {
    FTile x{};
    if constexpr (MODE == 2) {
        x.j0 = (t % P.npb) * kMaxN;
        t /= P.npb;
        x.i0 = (t % P.nkb) * 64;
        x.Ql = t / P.nkb;
    } else {
        const int per = P.nkb * P.npb;
        const int e = t / per, r = t - e * per;
        const int4 w = P.work[e];
        x.aD = w.x & 0xFFFF;
        x.bD = (int)((unsigned)w.x >> 16);
        x.dk = w.y;
        x.dn = w.z;
        x.n0 = w.w;
        x.kblk = r / P.npb;
        x.pblk = r - x.kblk * P.npb;
    }
    return x;
}

// Runs of P.run consecutive tiles, dealt round-robin to the blocks.
__device__ __forceinline__ int f_tile_of(const FParams& P, int i) {
    return ((i / P.run) * (int)gridDim.x + (int)blockIdx.x) * P.run + i % P.run;
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_digits(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ FParams P) {
    if (*P.flag) return;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int stage_bytes = kDig * (kAPlane + P.bplane);
    uint64_t* full = (uint64_t*)(smem + kStages * stage_bytes);   // [kStages]
    uint64_t* empty = full + kStages;                             // [kStages]
    uint64_t* tfull = empty + kStages;                            // [kDig]
    uint64_t* tempty = tfull + kDig;                              // [kDig]
    uint64_t* mdone = tempty + kDig;
    uint32_t* tmem_slot = (uint32_t*)(mdone + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    int* ebs = (int*)(smem + kStages * stage_bytes + 256);          // [4][kMaxN] column exponents
    double* bufs = (double*)(ebs + 4 * kMaxN);                       // [4][16][pb Nwex + 1] complex
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // rows of a stage that no box writes only feed accumulator entries that
    // are ignored; clear them once so that they hold finite values
    for (int i = threadIdx.x; i < kStages * stage_bytes / 16; i += blockDim.x)
        ((uint4*)smem)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int p = 0; p < kDig; ++p) {
            mbar_init(&tfull[p], 1);
            mbar_init(&tempty[p], kEpiWarps);
        }
        mbar_init(mdone, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t g = 0;
            bool ok = true;
            for (int it = 0; ok && !*abort_flag; ++it) {
                const int t = f_tile_of(P, it);
                if (t >= P.ntiles) break;
                const FTile x = f_tile<MODE>(P, t);
                const int bn = MODE == 2 ? 0 : (MODE == 0 ? x.n0 + x.dn : P.Nw2 - x.n0 - P.nb) + P.m0;
                for (int ch = 0; ch < P.nchunk; ++ch, ++g) {
                    const int s = g % kStages;
                    if (!mbar_wait(&empty[s], ((g / kStages) & 1) ^ 1, P.budget, abort_flag)) {
                        ok = false;
                        break;
                    }
                    uint8_t* st = smem + s * stage_bytes;
                    mbar_expect_tx(&full[s], P.txbytes);
                    for (int u = 0; u < kDig; ++u) {
                        uint8_t* sa = st + u * kAPlane;
                        uint8_t* sb = st + kDig * kAPlane + u * P.bplane;
                        if constexpr (MODE == 2) {
                            tma_load_4d(sa, &tmA, &full[s], P.jA[ch], 1 - P.cw[ch], x.i0, x.Ql * kDig + u);
                            tma_load_4d(sb, &tmB, &full[s], P.jB[ch], 1 + P.cw[ch], x.j0, x.Ql * kDig + u);
                        } else {
                            tma_load_5d(sa, &tmA, &full[s], P.jA[ch], 1 - P.cw[ch], x.n0, x.kblk * P.kb,
                                        x.aD * kDig + u);
                            tma_load_5d(sb, &tmB, &full[s], P.jB[ch], 1 + P.cw[ch], bn, x.pblk * P.pb,
                                        x.bD * kDig + u);
                        }
                    }
                }
            }
            // after an abort, wait (bounded) until the copies already issued have landed
            if (*abort_flag)
                for (uint32_t k = 0; k < (uint32_t)kStages && k < g; ++k)
                    mbar_drain(&full[(g - 1 - k) % kStages], ((g - 1 - k) / kStages) & 1, kDrainBudget);
        }
    } else if (warp == 1) {
        // the whole warp runs the loop (see elect_one): with one thread in it,
        // an MMA took 85 clocks to issue whatever its size, and that was the limit
        uint32_t g = 0, tl = 0;
        bool ok = true;
        for (int it = 0; ok; ++it, ++tl) {
            if (f_tile_of(P, it) >= P.ntiles) break;
            for (int ch = 0; ok && ch < P.nchunk; ++ch, ++g) {
                const int s = g % kStages;
                ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (g / kStages) & 1, P.budget, abort_flag));
                if (!ok) break;
                tc_fence_after();
                // descriptors differ in the address field alone (units of 16 bytes)
                const uint64_t da = sdesc_k64(smem_u32(smem + s * stage_bytes));
                const uint64_t db = da + (uint64_t)(kDig * kAPlane >> 4);
                const uint32_t bp = (uint32_t)P.bplane >> 4;
                const uint32_t acc0 = ch != 0;
                // one digit of A after the other, each against all its digits of B:
                // neighbouring MMAs go to different accumulators (back to back on one,
                // such small ones wait for each other), and the levels are complete
                // one by one
#pragma unroll
                for (int u = 0; u < kDig; ++u) {
                    if (u == 0 && ch == 0) {
                        for (int p = 0; ok && p < kDig; ++p)
                            ok = __all_sync(0xffffffffu, mbar_wait(&tempty[p], (tl & 1) ^ 1, P.budget, abort_flag));
                        if (!ok) break;
                        tc_fence_after();
                    }
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < 2; ++k)   // 16 values of K = 32 bytes
#pragma unroll
                            for (int v = 0; v < kDig - u; ++v)
                                mma_f16(tmem_base + (uint32_t)((u + v) * kMaxN), da + (uint64_t)(u * (kAPlane >> 4) + 2 * k),
                                        db + (uint64_t)(v * bp + 2 * k), P.idesc, (u | k) ? 1u : acc0);
                        if (ch == P.nchunk - 1) mma_commit(&tfull[u]);
                    }
                    __syncwarp();
                }
                if (ok && elect_one()) mma_commit(&empty[s]);
                __syncwarp();
            }
        }
        // wait (bounded) for every MMA this warp issued before tensor memory is freed
        if (elect_one()) mma_commit(mdone);
        __syncwarp();
        mbar_drain(mdone, 0, kDrainBudget);
    } else {
        const int quad = warp & 3;             // tensor-memory lane quarter of this warp
        const int part = (warp - 2) >> 2;      // its quarter of the columns
        const int row = quad * 32 + lane;
        const int c = row & 1, i = row >> 1;   // component of the result, row within the tile
        const int ncp = P.ncols / 4;           // columns of this warp (at most 16)
        const int col0 = part * ncp;
        const int n_l = MODE == 2 ? 0 : i % P.nb, k_l = MODE == 2 ? 0 : i / P.nb;
        const int rs = P.pb * P.Nwex + 1;      // entries of a row's buffer (odd: no bank conflicts)
        double* buf = bufs + (size_t)quad * 16 * rs * 2;
        int* eb = ebs + quad * kMaxN;
        const int pr = lane >> 1;
        // this thread's share of the quarter's stores and column exponents
        const int tq = part * 32 + lane;
        int ckp = 0, cn = 0;                   // column tq: momentum, frequency in the window
        uint32_t dstp[4] = {0, 0, 0, 0};       // per column: entry of the row's buffer, or 255
        if constexpr (MODE != 2) {
            ckp = tq / P.W;
            cn = tq - ckp * P.W;
            const int shift = MODE == 0 ? n_l : P.nb - 1 - n_l;   // window column of m = 0
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const int kp_l = (col0 + u) / P.W, m = col0 + u - kp_l * P.W - shift;
                const uint32_t dst = (u < ncp && kp_l < P.pb && m >= 0 && m < P.Nwex) ? kp_l * P.Nwex + m : 255;
                dstp[u >> 2] |= dst << (8 * (u & 3));
            }
        }
        // exponents of this thread's row and of column tq
        auto exps = [&](const FTile& x, int& eA, int& eC) {
            eA = eC = 0;
            if constexpr (MODE == 2) {
                if (x.i0 + i < P.N) eA = P.exA[(size_t)x.Ql * P.N + x.i0 + i];
                if (tq < kMaxN && x.j0 + tq < P.N) eC = P.exB[(size_t)x.Ql * P.N + x.j0 + tq];
            } else {
                const int k1 = x.kblk * P.kb + k_l, n1 = x.n0 + n_l;
                if (k1 < P.Nc && n1 < P.Nw2) eA = P.exA[(size_t)x.aD * P.N + k1 * P.Nw2 + n1];
                const int kp = x.pblk * P.pb + ckp;
                const int nn = (MODE == 0 ? x.n0 + x.dn : P.Nw2 - x.n0 - P.nb) + P.m0 + cn;
                if (ckp < P.pb && kp < P.Nc && nn >= 0 && nn < P.Nw2)
                    eC = P.exA[(size_t)x.bD * P.N + kp * P.Nw2 + nn];
            }
        };
        int t = f_tile_of(P, 0);
        int eA = 0, eC = 0;
        if (t < P.ntiles) exps(f_tile<MODE>(P, t), eA, eC);
        uint32_t tl = 0;
        for (int it = 0; t < P.ntiles; ++it, ++tl) {
            // sum of the levels, level p counting 2^(56-8p): (hi, mid, lo)
            uint32_t lo[16], mid[16], hi[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) lo[u] = mid[u] = hi[u] = 0u;
            bool fail = false;
#pragma unroll
            for (int p = 0; p < kDig; ++p) {
                if (!fail) fail = __any_sync(0xffffffffu, !mbar_wait(&tfull[p], tl & 1, P.budget, abort_flag));
                if (fail) continue;
                tc_fence_after();
                const uint32_t ta = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(p * kMaxN + col0);
#pragma unroll
                for (int u0 = 0; u0 < 16; u0 += 8) {   // eight at a time: registers
                    float v[8];
                    tmem_ld8(ta + u0, v);
                    tmem_wait_ld();
                    if (u0 == 8) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&tempty[p]);
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int u = u0 + k, w = __float2int_rn(v[k]);
                        switch (p) {
                            case 0: add_level<0>(lo[u], mid[u], hi[u], w); break;
                            case 1: add_level<1>(lo[u], mid[u], hi[u], w); break;
                            case 2: add_level<2>(lo[u], mid[u], hi[u], w); break;
                            case 3: add_level<3>(lo[u], mid[u], hi[u], w); break;
                            case 4: add_level<4>(lo[u], mid[u], hi[u], w); break;
                            case 5: add_level<5>(lo[u], mid[u], hi[u], w); break;
                            case 6: add_level<6>(lo[u], mid[u], hi[u], w); break;
                            default: add_level<7>(lo[u], mid[u], hi[u], w);
                        }
                    }
                }
            }
            // the tile's entry is decoded only now (registers), and the next one's
            // exponents are loaded while this one is stored
            const int tn = f_tile_of(P, it + 1);
            const FTile x = f_tile<MODE>(P, t);
            int eAn, eCn;
            exps(f_tile<MODE>(P, tn < P.ntiles ? tn : t), eAn, eCn);
            if (tq < kMaxN) eb[tq] = eC;
            // the previous tile's stores have read the buffer
            bulk_wait_read_all();
            if (quarter_any(quad, fail)) break;
            if constexpr (MODE == 2) {
                // lane pairs exchange components of two columns: 32 contiguous bytes of a row
                const int K1 = x.i0 + i;
                double2* dst = P.scr + ((size_t)x.Ql * P.N + K1) * P.N + x.j0 + col0 + c;
#pragma unroll
                for (int u = 0; u < 16; u += 2) {
                    const double v0 = fixed_to_f64(lo[u], mid[u], hi[u], eA + eb[col0 + u] - 68, false);
                    const double v1 = fixed_to_f64(lo[u + 1], mid[u + 1], hi[u + 1], eA + eb[col0 + u + 1] - 68, false);
                    const double y = __shfl_xor_sync(0xffffffffu, c ? v0 : v1, 1);
                    if (K1 < P.N && x.j0 + col0 + u + c < P.N) dst[u] = c ? make_double2(y, v1) : make_double2(v0, y);
                }
                quarter_any(quad, false);   // the exponents are read
            } else {
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const uint32_t dst = (dstp[u >> 2] >> (8 * (u & 3))) & 0xFFu;
                    const double val = fixed_to_f64(lo[u], mid[u], hi[u], eA + eb[col0 + u] - 68, MODE == 0);
                    if (dst != 255) buf[(pr * rs + dst) * 2 + c] = val;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                quarter_any(quad, false);
                for (int task = tq; task < 16 * P.pb; task += 128) {
                    const int sr = task & 15, kp_l = task >> 4, ii = quad * 16 + sr;
                    const int k1 = x.kblk * P.kb + ii / P.nb, n1 = x.n0 + ii % P.nb, n2 = n1 + x.dn;
                    const int kp = x.pblk * P.pb + kp_l;
                    if (ii >= P.kb * P.nb || k1 >= P.Nc || n1 >= P.Nw2 || n2 < 0 || n2 >= P.Nw2 || kp >= P.Nc)
                        continue;
                    const int k1y = k1 / P.Lx, k1x = k1 - k1y * P.Lx, dky = x.dk / P.Lx, dkx = x.dk - dky * P.Lx;
                    const int kpy = kp / P.Lx, kpx = kp - kpy * P.Lx;
                    int k2x = k1x + dkx, k2y = k1y + dky;
                    k2x -= k2x >= P.Lx ? P.Lx : 0;
                    k2y -= k2y >= P.Ly ? P.Ly : 0;
                    // q = kp (-) k2 (particle-hole) or kp (+) k1 (particle-particle)
                    int qx = MODE == 0 ? kpx - k2x : kpx + k1x, qy = MODE == 0 ? kpy - k2y : kpy + k1y;
                    if (MODE == 0) {
                        qx += qx < 0 ? P.Lx : 0;
                        qy += qy < 0 ? P.Ly : 0;
                    } else {
                        qx -= qx >= P.Lx ? P.Lx : 0;
                        qy -= qy >= P.Ly ? P.Ly : 0;
                    }
                    const int q = qx + P.Lx * qy;
                    const int mlim = MODE == 0 ? min(P.Nwex, min(P.Nw2 - n1, P.Nw2 - n2) - P.m0)
                                               : min(P.Nwex, min(n1, n2) + 1 - P.m0);
                    if (q >= P.Nkex || mlim <= 0) continue;
                    const int k2 = k2x + P.Lx * k2y;
                    bulk_add_f64(P.acc + ((size_t)(k1 * P.Nw2 + n1) * P.N + (size_t)(k2 * P.Nw2 + n2)) * P.NQ +
                                     (size_t)q * P.Nwex,
                                 (double2*)buf + sr * rs + kp_l * P.Nwex, (uint32_t)(16 * mlim));
                }
                bulk_commit();
            }
            t = tn;
            eA = eAn;
            eC = eCn;
        }
        bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) atomicOr(P.status, (unsigned)G4_DEV_TIMEOUT);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// acc[K1][K2][Q0 .. Q0+nQ) += scratch [ql][K1][K2]: runs of nQ entries per
// (K1, K2) staged in shared memory, one bulk reduction each.
constexpr int kMergeK2 = 64;
constexpr int kGroupQ = 16;

__global__ void __launch_bounds__(256) k_merge64(const double2* __restrict__ scr, double2* __restrict__ acc,
                                                 int Q0, int nQ, int N, int NQ,
                                                 const unsigned* __restrict__ flag) {
    if (*flag) return;
    __shared__ __align__(16) double2 run[kMergeK2 * (kGroupQ + 1)];
    const int K1 = blockIdx.y, K2b = blockIdx.x * kMergeK2;
    const int ld = nQ + 1;
    for (int t = threadIdx.x; t < nQ * kMergeK2; t += blockDim.x) {
        const int ql = t / kMergeK2, k2l = t - ql * kMergeK2;
        if (K2b + k2l < N) run[k2l * ld + ql] = scr[((size_t)ql * N + K1) * N + K2b + k2l];
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < kMergeK2) {
        const int K2 = K2b + threadIdx.x;
        if (K2 < N)
            bulk_add_f64(acc + ((size_t)K1 * N + K2) * NQ + Q0, run + threadIdx.x * ld, (uint32_t)(16 * nQ));
        bulk_commit();
        bulk_wait_read_all();
    }
}

// ------------------------------------------------------------------ host
struct F64Plan {
    double tiles = 0;          // exchange tiles of a batch
    int kb = 0, nb = 0, W = 0, pb = 0, nkb = 0, npb = 0, N = 0;
    int Jh = 0, J = 0, Bp = 0, gcap = 0, nQg = 0;
    std::vector<int> gd0, gdn, gw0, gwn;   // per group: diagonals, work entries
    int4* work = nullptr;
    int* pos0 = nullptr;
    __half* X = nullptr;
    int* ex = nullptr;
    __half* ab = nullptr;      // direct: [2][nQg * 8][N][3][Bp]
    int* exab = nullptr;       // [2][nQg][N]
    double2* scr = nullptr;    // [nQg][N][N]
    CUtensorMap mA, mB, dA, dB;
    int smem = 0, dsmem = 0;
    int sms = 0;
};

PFN_cuTensorMapEncodeTiled_v12000 f_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

// Shared memory of k_gemm_digits; entries: pb Nwex of a row's run buffer (0: direct).
int f_smem(int ncols, int entries) {
    return kStages * kDig * (kAPlane + ncols * 64) + 1024 + 256 + 4 * kMaxN * 4 + 4 * 16 * (entries + 1) * 16;
}

bool encode_maps(const G4Dims& d, F64Plan& X) {
    auto enc = f_encoder();
    if (!enc) return false;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    auto make = [&](CUtensorMap* m, int rank, void* base, const cuuint64_t* dims, const cuuint64_t* str,
                    const cuuint32_t* box) {
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, rank, base, dims, str, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    const cuuint64_t J = X.J, Nw2 = d.Nw2, Nc = d.Nc;
    const cuuint64_t xd[5] = {J, 3, Nw2, Nc, (cuuint64_t)X.gcap * kDig};
    const cuuint64_t xs[4] = {J * 2, J * 6, J * 6 * Nw2, J * 6 * Nw2 * Nc};
    const cuuint32_t ba[5] = {kChunk, 2, (cuuint32_t)X.nb, (cuuint32_t)X.kb, 1};
    const cuuint32_t bb[5] = {kChunk, 1, (cuuint32_t)X.W, (cuuint32_t)X.pb, 1};
    if (!make(&X.mA, 5, X.X, xd, xs, ba) || !make(&X.mB, 5, X.X, xd, xs, bb)) return false;
    if (!X.ab) return true;
    const cuuint64_t B = X.Bp, N = d.N;
    const cuuint64_t dd[4] = {B, 3, N, (cuuint64_t)X.nQg * kDig};
    const cuuint64_t ds[3] = {B * 2, B * 6, B * 6 * N};
    const cuuint32_t da[4] = {kChunk, 2, 64, 1}, db[4] = {kChunk, 1, kMaxN, 1};
    __half* bside = X.ab + (size_t)X.nQg * kDig * d.N * 3 * X.Bp;
    return make(&X.dA, 4, X.ab, dd, ds, da) && make(&X.dB, 4, bside, dd, ds, db);
}

// Clocks of one exchange tile of N columns and nsteps x 16 values of K: measured
// over shapes of one to 256 sites and 2 to 128 frequencies, within a tenth.
double tile_clocks(int N, int nsteps) { return 8000.0 + 10.5 * nsteps * (kARows + N); }

// The tile shape (kb x nb rows, pb x W columns) with the least time over all
// diagonals.
bool choose_tile(const G4Dims& d, int nsteps, F64Plan& X) {
    double best = 1e300;
    for (int nb = 1; nb <= 16 && nb <= d.Nw2; ++nb) {
        const int W = nb + d.Nwex - 1;
        if (W > kMaxN) break;
        double blocks = 0;
        for (int dn = -(d.Nw2 - 1); dn < d.Nw2; ++dn) blocks += (d.Nw2 - std::abs(dn) + nb - 1) / nb;
        for (int kb = 1; kb <= d.Nc && 2 * kb * nb <= kARows; ++kb)
            for (int pb = 1; pb <= d.Nc; ++pb) {
                const int N = (W * pb + 15) / 16 * 16;
                if (N > kMaxN || f_smem(N, pb * d.Nwex) > kMaxSmem) break;
                const int nkb = (d.Nc + kb - 1) / kb, npb = (d.Nc + pb - 1) / pb;
                const double cost = blocks * nkb * npb * tile_clocks(N, nsteps);
                if (cost < best) {
                    best = cost;
                    X.kb = kb;
                    X.nb = nb;
                    X.W = W;
                    X.pb = pb;
                    X.nkb = nkb;
                    X.npb = npb;
                    X.N = N;
                    X.tiles = blocks * nkb * npb * d.Nc;
                }
            }
    }
    return best < 1e300;
}

void f_free(F64Plan* X) {
    void* ptrs[] = {X->work, X->pos0, X->X, X->ex, X->ab, X->exab, X->scr};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete X;
}

// Device memory the plan may take (the operands of a batch are formed in groups
// of diagonals that fit): by the problem's sizes alone, as much as the
// accumulator and the staged G take, at least 512 MB and at most 4 GB.  One batch
// of 64 on the 4x4 cluster with 64 frequencies and 8 x 16 transfers takes 20.7
// ms with 4 GB (four groups), 20.1 with 8 (two), 21.4 with 2, 22.4 with 1.
size_t plan_bytes(const G4Dims& d, int batch) {
    const size_t held = ((size_t)d.E + (size_t)batch * 2 * d.N * d.N) * sizeof(double2);
    return std::min<size_t>(std::max<size_t>(held, (size_t)512 << 20), (size_t)4 << 30);
}

// Whether a batch of `staged` measurements takes less time here than in the plain
// kernels, by times measured on the shapes of tile_clocks and 4 to 64
// measurements: the work here does not shrink with the transfer momenta (every
// tile holds all of them) nor, below 16 measurements, with the batch.  In
// microseconds; where the two sides are not near each other the estimates are
// within a quarter.  (By the number of element-updates alone, from 4e6 on, 16x16
// sites with 2 frequencies and 4 momenta took 2.7 ms for 16 measurements, 0.9 in
// the plain kernel.)
bool faster_here(const G4Dims& d, const F64Plan& X, int staged, int sms, size_t ngroups) {
    const double N2 = (double)d.N * d.N;
    const int live = X.Jh > 16 ? (staged + 31) / 32 * 32 : 16;
    const double exchange = 30.0 + X.tiles / sms * tile_clocks(X.N, live / 4) / 1900.0;
    // the check and the pack: G read twice, digits written; TB/s
    const double rate = 3.6 * d.Nw2 / (d.Nw2 + 3.0) / (ngroups == 1 ? 1.0 : d.Nw2 < 24 ? 1.6 : 1.2);
    const double pack = 20.0 + N2 * (64.0 * staged + 96.0 * live) / rate * 1e-6;
    double direct = 0.0;
    if (has_direct(d.ch))
        direct = 25.0 * ((d.NQ + X.nQg - 1) / X.nQg) + d.NQ * N2 * (12.0 + 0.4 * staged) * 1e-6;
    return exchange + pack + direct < 5.0 + (double)d.E * staged * update_fp64_ps(d) * 1e-6;
}

}  // namespace

void f64tc_prepare(g4_ctx* h) {
    const G4Dims& d = h->d;
    // a memory limit or a wait budget of the caller's is kept as it was
    if (h->opt.mem_limit > 0 || h->opt.timeout_cycles > 0 || d.Nwex > kMaxWex) return;
    F64Plan* X = new (std::nothrow) F64Plan();
    if (!X) return;
    const bool cross = d.ch == G4_PH_TRANSVERSE || d.ch == G4_PP_UPDOWN;
    const int pad = cross ? 32 : 16;   // a spin's chunks of 32 when the spins are exchanged
    X->Jh = (h->batch + pad - 1) / pad * pad;
    if (X->Jh > 16) X->Jh = (X->Jh + 31) / 32 * 32;
    X->J = 2 * X->Jh;
    X->Bp = (h->batch + 31) / 32 * 32;
    std::vector<int2> dl;
    std::vector<int> itemlen;
    diag_list(d, dl, itemlen);
    bool ok = choose_tile(d, X->J / 8, *X);
    const size_t budget = plan_bytes(d, h->batch);
    // direct term: transfers per group, whose scratch stays in L2 where it can
    size_t direct_b = 0;
    if (has_direct(d.ch)) {
        const size_t one = (size_t)d.N * d.N * sizeof(double2);
        X->nQg = (int)std::min<size_t>(std::min(kGroupQ, d.NQ), std::max<size_t>(4, ((size_t)64 << 20) / one));
        const size_t per_Q = one + (size_t)2 * d.N * (3 * X->Bp * kDig * sizeof(__half) + sizeof(int));
        X->nQg = (int)std::min<size_t>(std::min(X->nQg, d.NQ), std::max<size_t>(1, budget / 2 / per_Q));
        direct_b = X->nQg * per_Q;
    }
    const size_t per_diag = (size_t)d.N * (3 * X->J * kDig * sizeof(__half) + sizeof(int));
    ok = ok && budget > direct_b && (budget - direct_b) / per_diag >= 2;
    if (ok) {
        const size_t fit = std::min<size_t>((budget - direct_b) / per_diag, 65535);
        const size_t ng = (dl.size() + fit - 1) / fit;
        X->gcap = (int)std::min<size_t>(fit, ((dl.size() + ng - 1) / ng + 1) / 2 * 2);
        ok = ok && (size_t)X->gcap * kDig < ((size_t)1 << 31) &&
             cudaDeviceGetAttribute(&X->sms, cudaDevAttrMultiProcessorCount, h->device) == cudaSuccess &&
             faster_here(d, *X, h->batch, X->sms, ng);
    }
    std::vector<int4> work;
    std::vector<int> pos0(d.Nc, -1);
    if (ok) {
        for (size_t p = 0; p < dl.size(); ++p)
            if (dl[p].y == 0) pos0[dl[p].x] = (int)p;
        int pos = 0;
        for (size_t it = 0; it < itemlen.size();) {
            const int g0 = pos, w0 = (int)work.size();
            while (it < itemlen.size() && pos + itemlen[it] - g0 <= X->gcap) {
                const int len = itemlen[it];
                for (int u = 0; u < len; ++u) {
                    const int a = pos + u - g0, b = len == 2 ? pos + (1 - u) - g0 : a;
                    const int dk = dl[pos + u].x, dn = dl[pos + u].y;
                    const int nlo = std::max(0, -dn), nhi = std::min(d.Nw2, d.Nw2 - dn);
                    for (int n0 = nlo; n0 < nhi; n0 += X->nb) work.push_back(make_int4(a | (b << 16), dk, dn, n0));
                }
                pos += len;
                ++it;
            }
            X->gd0.push_back(g0);
            X->gdn.push_back(pos - g0);
            X->gw0.push_back(w0);
            X->gwn.push_back((int)work.size() - w0);
        }
    }
    size_t held = 0;
    auto get = [&](void** p, size_t bytes) {
        if (ok && cudaMalloc(p, bytes) != cudaSuccess) {
            cudaGetLastError();
            *p = nullptr;
            ok = false;
        }
        if (ok) held += bytes;
    };
    get((void**)&X->work, work.size() * sizeof(int4));
    get((void**)&X->pos0, (size_t)d.Nc * sizeof(int));
    get((void**)&X->X, (size_t)X->gcap * kDig * d.N * 3 * X->J * sizeof(__half));
    get((void**)&X->ex, (size_t)X->gcap * d.N * sizeof(int));
    if (has_direct(d.ch)) {
        get((void**)&X->ab, (size_t)2 * X->nQg * kDig * d.N * 3 * X->Bp * sizeof(__half));
        get((void**)&X->exab, (size_t)2 * X->nQg * d.N * sizeof(int));
        get((void**)&X->scr, (size_t)X->nQg * d.N * d.N * sizeof(double2));
    }
    // exponents of off-grid rows are read and ignored
    ok = ok && cudaMemset(X->ex, 0, (size_t)X->gcap * d.N * sizeof(int)) == cudaSuccess &&
         cudaMemcpy(X->work, work.data(), work.size() * sizeof(int4), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(X->pos0, pos0.data(), pos0.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess &&
         encode_maps(d, *X) && raise_smem_limit(k_spread) == cudaSuccess && raise_smem_limit(k_gemm_digits<0>) == cudaSuccess &&
         raise_smem_limit(k_gemm_digits<1>) == cudaSuccess && raise_smem_limit(k_gemm_digits<2>) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        f_free(X);
        return;
    }
    X->smem = std::max(kMinSmem, f_smem(X->N, X->pb * d.Nwex));
    X->dsmem = std::max(kMinSmem, f_smem(kMaxN, 0));
    h->bytes += held;
    h->f64tc = X;
}

void f64tc_release(g4_ctx* h) {
    if (h->f64tc) f_free((F64Plan*)h->f64tc);
    h->f64tc = nullptr;
}

bool f64tc_wanted(const g4_ctx* h, int staged) {
    // fewer than four measurements: k_spread has no quarter to spare
    if (!h->f64tc || h->f64_plain || staged < 4) return false;
    const F64Plan* X = (const F64Plan*)h->f64tc;
    if (staged < h->batch && !faster_here(h->d, *X, staged, X->sms, X->gd0.size())) return false;
    // the sign factors must stay in the digits' exponent range
    for (int r = 0; r < staged; ++r) {
        const double a = std::fabs(h->slot_sign[r]);
        if (a != 0.0 && !(a > 1e-12 && a < 1e12)) return false;
    }
    return true;
}

g4_status f64tc_run(g4_ctx* h, int staged) {
    const F64Plan* X = (const F64Plan*)h->f64tc;
    const G4Dims& d = h->d;
    unsigned* flag = h->gmax;
    FSigns sg{};
    SpreadArgs sp{};
    for (int r = 0; r < staged; ++r) {
        sg.rs[r] = std::sqrt(std::fabs(h->slot_sign[r]));
        sg.neg[r] = h->slot_sign[r] < 0.0;
        sp.se[r] = sg.rs[r] > 0.0 ? (signed char)std::ilogb(sg.rs[r]) : (signed char)-128;
    }
    FParams P{};
    P.acc = h->acc;
    P.status = h->dstatus;
    P.flag = flag;
    P.Lx = d.Lx;
    P.Ly = d.Ly;
    P.Nc = d.Nc;
    P.Nw2 = d.Nw2;
    P.N = d.N;
    P.Nwex = d.Nwex;
    P.Nkex = d.Nkex;
    P.NQ = d.NQ;
    P.m0 = d.m0;
    P.kb = X->kb;
    P.nb = X->nb;
    P.W = X->W;
    P.pb = X->pb;
    P.nkb = X->nkb;
    P.npb = X->npb;
    P.ncols = X->N;
    P.bplane = X->N * 64;
    P.txbytes = (uint32_t)(kDig * 64 * (2 * X->nb * X->kb + X->W * X->pb));
    P.idesc = idesc_f16(kARows, X->N);
    P.budget = 4000000000LL;
    // chunks of K that hold staged measurements (a batch of at most 16 has both
    // spins in one chunk)
    const int live = X->Jh > 16 ? (staged + 31) / 32 * 32 : 16;
    const bool cross = d.ch == G4_PH_TRANSVERSE || d.ch == G4_PP_UPDOWN;
    auto chunk = [&](int ja, int jb) {
        for (int w = 0; w < 2; ++w, ++P.nchunk) {
            P.jA[P.nchunk] = ja;
            P.jB[P.nchunk] = jb;
            P.cw[P.nchunk] = w;
        }
    };
    if (X->Jh <= 16) {
        chunk(0, 0);
    } else {
        for (int sp = 0; sp < 2; ++sp)
            for (int u = 0; u < live; u += 32) chunk((cross ? 1 - sp : sp) * X->Jh + u, sp * X->Jh + u);
    }
    const int njb = (d.Nw2 + kPackJ - 1) / kPackJ;
    cudaError_t e;
    prof_begin(h, G4_K_PACK_EXCHANGE);
    const bool direct = has_direct(d.ch);
    const size_t ssm = (size_t)(direct ? 3 : 2) * staged * 256 * sizeof(unsigned short);
    const long long sblocks = ((long long)d.N * d.N + 255) / 256;
    k_spread<<<(int)std::min<long long>(sblocks, 16LL * X->sms), 256, ssm, h->stream>>>(h->Gfull, staged, sp, direct, d,
                                                                                       flag);
    prof_end(h, G4_K_PACK_EXCHANGE);
    if ((e = cudaGetLastError()) != cudaSuccess) return g4_cuda_fail(h, e, "digit spread launch");
    for (size_t g = 0; g < X->gd0.size(); ++g) {
        prof_begin(h, G4_K_PACK_EXCHANGE);
        // |dn| of the group's first and last diagonal (see diag_pos)
        auto dn_of = [&](int pos) { return pos < d.Nc ? 0 : (pos - d.Nc) / (2 * d.Nc) + 1; };
        const int dn0 = dn_of(X->gd0[g]), dn1 = dn_of(X->gd0[g] + X->gdn[g] - 1);
        const int nband = std::min(njb, (dn1 - dn0) / kPackJ + 2);
        k_pack_digits<<<dim3(d.Nc * 2 * nband, d.N), 256, kPackJ * 2 * (X->J + 2) * sizeof(double), h->stream>>>(
            h->Gfull, staged, X->Jh, live, sg, X->pos0, X->gd0[g], X->gdn[g], dn0, dn1, nband, X->X, X->ex, d, flag);
        prof_end(h, G4_K_PACK_EXCHANGE);
        if ((e = cudaGetLastError()) != cudaSuccess) return g4_cuda_fail(h, e, "digit pack launch");
        P.work = X->work + X->gw0[g];
        P.exA = X->ex;
        const int per = X->nkb * X->npb;
        P.ntiles = X->gwn[g] * per;
        // consecutive tiles share operand rows: a run of two row blocks, unless
        // that would leave SMs without one
        P.run = std::max(1, std::min(2 * per, P.ntiles / (8 * X->sms)));
        const int grid = std::min((P.ntiles + P.run - 1) / P.run, X->sms);
        prof_begin(h, G4_K_EXCHANGE);
        auto* kern = d.ch == G4_PP_UPDOWN ? k_gemm_digits<1> : k_gemm_digits<0>;
        kern<<<grid, kThreads, X->smem, h->stream>>>(X->mA, X->mB, P);
        prof_end(h, G4_K_EXCHANGE);
        if ((e = cudaGetLastError()) != cudaSuccess) return g4_cuda_fail(h, e, "digit exchange launch");
    }
    if (!direct) return G4_OK;
    P.scr = X->scr;
    P.exA = X->exab;
    P.exB = X->exab + (size_t)X->nQg * d.N;
    P.nkb = (d.N + 63) / 64;
    P.npb = (d.N + kMaxN - 1) / kMaxN;
    P.ncols = kMaxN;
    P.bplane = kMaxN * 64;
    P.txbytes = (uint32_t)(kDig * 64 * (128 + 64));
    P.idesc = idesc_f16(kARows, kMaxN);
    P.nchunk = 0;
    for (int u = 0; u < staged; u += 32) chunk(u, u);
    for (int Q0 = 0; Q0 < d.NQ; Q0 += X->nQg) {
        const int nQ = std::min(X->nQg, d.NQ - Q0);
        prof_begin(h, G4_K_DIRECT_SPLIT);
        k_pack_digits_ab<<<dim3(d.Nc * njb, nQ, 2), 256, kPackJ * 2 * (X->Bp + 2) * sizeof(double), h->stream>>>(
            h->Gfull, staged, X->Bp, (staged + 31) / 32 * 32, sg, Q0, X->nQg, X->ab, X->exab, d, flag);
        prof_end(h, G4_K_DIRECT_SPLIT);
        if ((e = cudaGetLastError()) != cudaSuccess) return g4_cuda_fail(h, e, "direct digit pack launch");
        P.ntiles = nQ * P.nkb * P.npb;
        P.run = std::max(1, std::min(4, P.ntiles / (8 * X->sms)));
        const int grid = std::min((P.ntiles + P.run - 1) / P.run, X->sms);
        prof_begin(h, G4_K_DIRECT);
        k_gemm_digits<2><<<grid, kThreads, X->dsmem, h->stream>>>(X->dA, X->dB, P);
        prof_end(h, G4_K_DIRECT);
        if ((e = cudaGetLastError()) != cudaSuccess) return g4_cuda_fail(h, e, "direct digit launch");
        prof_begin(h, G4_K_DIRECT_MERGE);
        k_merge64<<<dim3((d.N + kMergeK2 - 1) / kMergeK2, d.N), 256, 0, h->stream>>>(X->scr, h->acc, Q0, nQ, d.N,
                                                                                     d.NQ, flag);
        prof_end(h, G4_K_DIRECT_MERGE);
        if ((e = cudaGetLastError()) != cudaSuccess) return g4_cuda_fail(h, e, "direct digit merge launch");
    }
    return G4_OK;
}
