// Element-wise and layout kernels of the G4 path:
//   * G build, G = G0 d - G0 M G0 (Sec. 2), in the natural layout (FP64 path,
//     standalone g4_build_G) and in the diagonal-major complex64 layout the
//     mixed path consumes;
//   * the plain FP64 update of G4 with a batch of measurements (the
//     accumulation of Eq. (1), Sec. 2.1);
//   * the final normalisation by the sign sum and the transpose to the
//     exported layout.
#include <algorithm>
#include <type_traits>

#include "g4_gtilde.cuh"
#include "g4_internal.h"
#include "g4_ptx.cuh"

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// G[sp][i][j] = G0[sp][i] d_ij - G0[sp][i] M[sp][i][j] G0[sp][j], FP64.  A
// block takes kBuildU blocks of columns of one row (no division per entry,
// kBuildU independent loads in flight); FLAG: see launch_build_G_fp64, tested on
// the exponent fields.  Bound by the FP64 pipe and, with the test, the issue
// slots: 20 builds of N = 1000 took 0.95 ms with one entry per thread, 1.00 with
// the test always made and four, 0.83 with two and the test where it is used.
constexpr int kBuildU = 2;

template <bool M64, bool FLAG>
__global__ void __launch_bounds__(256) k_build_G_fp64(const void* __restrict__ M,
                                                      const double2* __restrict__ G0,
                                                      double2* __restrict__ G, int N,
                                                      unsigned* __restrict__ flag) {
    using MV = typename std::conditional<M64, float2, double2>::type;
    bool bad = false;
    const int j0 = blockIdx.x * (kBuildU * blockDim.x) + threadIdx.x;
    for (int row = blockIdx.y; row < 2 * N; row += gridDim.y) {
        const int sp = row >= N ? 1 : 0, i = row - sp * N;
        const double2 gi = G0[row], ngi = make_double2(-gi.x, -gi.y);
        const MV* mrow = reinterpret_cast<const MV*>(M) + (size_t)row * N;
        MV m[kBuildU];
        double2 gj[kBuildU];
#pragma unroll
        for (int u = 0; u < kBuildU; ++u) {
            const int j = j0 + u * blockDim.x;
            if (j < N) {
                m[u] = mrow[j];
                gj[u] = G0[sp * N + j];
            }
        }
#pragma unroll
        for (int u = 0; u < kBuildU; ++u) {
            const int j = j0 + u * blockDim.x;
            if (j >= N) break;
            double2 v = cmul(cmul(ngi, make_double2(m[u].x, m[u].y)), gj[u]);
            if (i == j) v = make_double2(v.x + gi.x, v.y + gi.y);
            G[(size_t)row * N + j] = v;
            if constexpr (!FLAG) continue;
            // off the FP64 pipe
            const long long bx = __double_as_longlong(v.x) & 0x7FFFFFFFFFFFFFFFll;
            const long long by = __double_as_longlong(v.y) & 0x7FFFFFFFFFFFFFFFll;
            constexpr unsigned lo = (unsigned)(1023 - kF64tcExp) << 20, span = (unsigned)(2 * kF64tcExp) << 20;
            bad = bad || ((unsigned)(bx >> 32) - lo > span && bx != 0) ||
                  ((unsigned)(by >> 32) - lo > span && by != 0);
        }
    }
    if (FLAG && bad) *flag = 1u;
}

// The staged measurements' FP64 update of every accumulator entry, for channel
// CH (see g4.h).  Block row K1 = blockIdx.y; groups of RS lanes run over (K2, Q)
// with Q fastest, so the accumulator read-modify-write, once per batch, is
// coalesced; the lanes of a group share out the measurements and add up their
// sums by shuffles.  The kernel of shapes the tiled one does not take (RS = 1,
// measurement by measurement onto the accumulator: sums apart from it are two
// more operations on the FP64 pipe, which bounds the kernel; one measurement at a
// time on the 4x4 cluster with 32 frequencies, particle-particle, 0.25 ms with
// them, 0.22 without) and of small problems, where a lane's chain over the
// measurements is the whole time (1024 entries, 16 measurements: 29 us with RS =
// 1, 5 with 16).
template <int CH, int RS>
__global__ void k_update_fp64(const double2* __restrict__ Gb, const __grid_constant__ G4Signs signs,
                              int staged, double2* __restrict__ acc, const int* __restrict__ kadd,
                              const int* __restrict__ ksub, G4Dims d,
                              const unsigned* __restrict__ only_if) {
    if (only_if && !*only_if) return;
    const int K1 = blockIdx.y;
    const int k1 = K1 / d.Nw2, n1 = K1 - k1 * d.Nw2;
    const size_t NN = (size_t)d.N * d.N;
    const int per = d.N * d.NQ;
    double2* row = acc + (size_t)K1 * per;
    const int sub = threadIdx.x % RS, step = gridDim.x * (blockDim.x / RS);
    // a warp's lanes stay together to the end (the shuffles take all of them)
    const int first = blockIdx.x * (blockDim.x / RS) + threadIdx.x / RS;
    for (int base = first - (int)(threadIdx.x & 31) / RS; base < per; base += step) {
        const int idx0 = base + (int)(threadIdx.x & 31) / RS, idx = min(idx0, per - 1);
        const int K2 = idx / d.NQ, Qi = idx - K2 * d.NQ;
        const int q = Qi / d.Nwex, m = d.m0 + Qi - q * d.Nwex;   // m: the transfer frequency
        const int k2 = K2 / d.Nw2, n2 = K2 - k2 * d.Nw2;
        double2 o = make_double2(0.0, 0.0);
        if (RS == 1 && idx0 < per) o = row[idx];
        for (int r = sub; r < staged; r += RS) {
            const double2* G = Gb + (size_t)(2 * r) * NN;
            const double sign = signs.s[r];
            double2 term = make_double2(0, 0);
            if (CH == G4_PP_UPDOWN) {
                // G_s(Q-K2, Q-K1) G_-s(K2, K1); Q-K has frequency index m + Nw2-1 - n
                const int f1 = m + d.Nw2 - 1 - n1, f2 = m + d.Nw2 - 1 - n2;
                if (f1 >= 0 && f1 < d.Nw2 && f2 >= 0 && f2 < d.Nw2) {
                    const int QK1 = ksub[q * d.Nc + k1] * d.Nw2 + f1;
                    const int QK2 = ksub[q * d.Nc + k2] * d.Nw2 + f2;
#pragma unroll
                    for (int sp = 0; sp < 2; ++sp) {
                        const double2 t = cmul(G[sp * NN + (size_t)QK2 * d.N + QK1],
                                               G[(1 - sp) * NN + (size_t)K2 * d.N + K1]);
                        term.x += t.x;
                        term.y += t.y;
                    }
                }
            } else {
                // an entry off the grid stays zero
                if (n1 + m >= d.Nw2 || n2 + m >= d.Nw2) break;
                const int K1Q = kadd[k1 * d.Nc + q] * d.Nw2 + n1 + m;
                const int K2Q = kadd[k2 * d.Nc + q] * d.Nw2 + n2 + m;
                double2 a = make_double2(0, 0), b = make_double2(0, 0), ex = make_double2(0, 0);
#pragma unroll
                for (int sp = 0; sp < 2; ++sp) {
                    const double2* g = G + sp * NN;
                    const double wgt = (CH == G4_PH_MAGNETIC && sp) ? -1.0 : 1.0;
                    if (CH != G4_PH_TRANSVERSE) {
                        double2 t = g[(size_t)K1Q * d.N + K1];
                        a.x += wgt * t.x;
                        a.y += wgt * t.y;
                        t = g[(size_t)K2 * d.N + K2Q];
                        b.x += wgt * t.x;
                        b.y += wgt * t.y;
                    }
                    // transverse pairs the opposite spin in the G(K2,K1) factor
                    const double2* gx = CH == G4_PH_TRANSVERSE ? G + (1 - sp) * NN : g;
                    const double2 t = cmul(gx[(size_t)K2 * d.N + K1], g[(size_t)K1Q * d.N + K2Q]);
                    ex.x += t.x;
                    ex.y += t.y;
                }
                const double2 ab = cmul(a, b);
                term = make_double2(ab.x - ex.x, ab.y - ex.y);
            }
            o.x += sign * term.x;
            o.y += sign * term.y;
        }
#pragma unroll
        for (int w = RS / 2; w > 0; w >>= 1) {
            o.x += __shfl_xor_sync(0xffffffffu, o.x, w);
            o.y += __shfl_xor_sync(0xffffffffu, o.y, w);
        }
        if (sub == 0 && idx0 < per) row[idx] = RS == 1 ? o : make_double2(row[idx].x + o.x, row[idx].y + o.y);
    }
}

// The same FP64 update for the particle-hole channels, tiled: a block owns a
// momentum pair (k1, k2) and a 16 x 16 tile of frequencies (n1, n2), one thread
// per (n1, n2), and walks the transfer momenta q and, inside, the staged
// measurements.  For each it stages in shared memory what the tile's products
// read -- the window of the G blocks (k1 (+) q, k2 (+) q) at rows n1 + m and
// columns n2 + m (exchange factor), the spin-weighted band G(K1+Q, K1) (a) and
// G(K2, K2+Q) (b), the G(K2, K1) tile -- and each thread sums its Nwex <= WX
// transfers in registers: the accumulator is read and written once per batch,
// and the sign rides on a and the G(K2, K1) tile, so that an element-update is
// fourteen operations.  Bound by the FP64 pipe (two lanes per clock and SM): one
// batch of 16 on the 4x4 cluster with 32 frequencies, 8 transfers and 4 momenta
// 3.75 ms, 4.78 in per-measurement launches of eighteen operations.  A
// measurement's products are summed before they meet the batch's sum: with all in
// one chain of twelve fused multiply-adds (3.13 ms) the error of a batch of 64
// against exact sums was 2.9e-16 of the products' moduli, 1.2e-16 so (and in
// per-measurement launches).
constexpr int kTileF = 16;      // frequencies per tile side
constexpr int kTileWex = 16;    // largest Nwex of the tiled form

__device__ __forceinline__ void cfma(double2& t, double2 a, double2 b) {
    t.x = fma(a.x, b.x, t.x);
    t.y = fma(a.x, b.y, t.y);
    t.x = fma(-a.y, b.y, t.x);
    t.y = fma(a.y, b.x, t.y);
}

template <int CH, int WXM>
__global__ void __launch_bounds__(kTileF * kTileF) k_update_fp64_tiled(
    const double2* __restrict__ Gb, const __grid_constant__ G4Signs signs, int staged,
    double2* __restrict__ acc, const int* __restrict__ kadd, G4Dims d,
    const unsigned* __restrict__ only_if) {
    if (only_if && !*only_if) return;
    extern __shared__ double2 sm[];
    const int Nw2 = d.Nw2, N = d.N, Nwex = d.Nwex;
    const int nt = (Nw2 + kTileF - 1) / kTileF;
    const int k1 = blockIdx.y / d.Nc, k2 = blockIdx.y - (blockIdx.y / d.Nc) * d.Nc;
    const int n1_0 = (blockIdx.x / nt) * kTileF, n2_0 = (blockIdx.x % nt) * kTileF;
    const int t1 = threadIdx.x / kTileF, t2 = threadIdx.x % kTileF;
    const int n1 = n1_0 + t1, n2 = n2_0 + t2;
    const bool live = n1 < Nw2 && n2 < Nw2;
    const size_t NN = (size_t)N * N;
    const int WX = kTileF + Nwex - 1;                // window side
    double2* X2 = sm;                                // [2 spins][WX][WX + 1]
    double2* X1 = X2 + 2 * WX * (WX + 1);            // [2 spins][kTileF t2][kTileF + 1 t1]
    double2* A = X1 + 2 * kTileF * (kTileF + 1);     // [kTileF t1][Nwex]
    double2* B = A + kTileF * Nwex;                  // [kTileF t2][Nwex]
    const double w1 = CH == G4_PH_MAGNETIC ? -1.0 : 1.0;  // weight of spin -1 in a, b
    for (int q = 0; q < d.Nkex; ++q) {
        const int k1q = kadd[k1 * d.Nc + q], k2q = kadd[k2 * d.Nc + q];
        double2* row = acc + ((size_t)(k1 * Nw2 + n1) * N + k2 * Nw2 + n2) * d.NQ + (size_t)q * Nwex;
        double2 sum[WXM];   // a single measurement goes onto the accumulator itself
#pragma unroll
        for (int m = 0; m < WXM; ++m)
            sum[m] = staged == 1 && m < Nwex && n1 + d.m0 + m < Nw2 && n2 + d.m0 + m < Nw2 ? row[m]
                                                                                          : make_double2(0.0, 0.0);
        for (int r = 0; r < staged; ++r) {
            const double2* G = Gb + (size_t)(2 * r) * NN;
            const double sign = signs.s[r];
            __syncthreads();  // the previous tiles are no longer read
            // G(K2, K1) of the tile (the transverse channel pairs the opposite spin);
            // a single measurement's stays over the transfers
            if (staged > 1 || q == 0)
            for (int t = threadIdx.x; t < 2 * kTileF * kTileF; t += blockDim.x) {
                const int sp = t / (kTileF * kTileF), u = t % (kTileF * kTileF);
                const int a2 = u / kTileF, a1 = u % kTileF;
                const int m1 = n1_0 + a1, m2 = n2_0 + a2;
                const int gs = CH == G4_PH_TRANSVERSE ? 1 - sp : sp;
                double2 v = make_double2(0.0, 0.0);
                if (m1 < Nw2 && m2 < Nw2) v = G[gs * NN + (size_t)(k2 * Nw2 + m2) * N + k1 * Nw2 + m1];
                X1[(sp * kTileF + a2) * (kTileF + 1) + a1] = make_double2(-sign * v.x, -sign * v.y);
            }
            for (int t = threadIdx.x; t < 2 * WX * WX; t += blockDim.x) {
                const int sp = t / (WX * WX), u = t % (WX * WX);
                const int i = u / WX, j = u % WX;
                const int f1 = n1_0 + i + d.m0, f2 = n2_0 + j + d.m0;  // frequencies n + m
                X2[(sp * WX + i) * (WX + 1) + j] =
                    (f1 < Nw2 && f2 < Nw2) ? G[sp * NN + (size_t)(k1q * Nw2 + f1) * N + k2q * Nw2 + f2]
                                           : make_double2(0.0, 0.0);
            }
            if (CH != G4_PH_TRANSVERSE) {
                for (int t = threadIdx.x; t < 2 * kTileF * Nwex; t += blockDim.x) {
                    const int side = t / (kTileF * Nwex), w = t % (kTileF * Nwex);
                    const int u = w / Nwex, m = w % Nwex;
                    const int mg = d.m0 + m;
                    double2 v = make_double2(0.0, 0.0);
                    // a(n1, m) = sum_s w_s G_s((k1 (+) q, n1 + m), (k1, n1)),
                    // b(n2, m) = sum_s w_s G_s((k2, n2), (k2 (+) q, n2 + m))
                    const int nn = (side ? n2_0 : n1_0) + u;
                    if (nn < Nw2 && nn + mg < Nw2) {
                        const size_t i0 = side ? (size_t)(k2 * Nw2 + nn) * N + k2q * Nw2 + nn + mg
                                               : (size_t)(k1q * Nw2 + nn + mg) * N + k1 * Nw2 + nn;
                        const double2 g0 = G[i0], g1 = G[NN + i0];
                        const double f = side ? 1.0 : sign;
                        v = make_double2(f * (g0.x + w1 * g1.x), f * (g0.y + w1 * g1.y));
                    }
                    (side ? B : A)[w] = v;
                }
            }
            __syncthreads();
#pragma unroll
            for (int m = 0; m < WXM; ++m) {
                if (m >= Nwex) break;
                double2 t = cmul(X1[t2 * (kTileF + 1) + t1], X2[(t1 + m) * (WX + 1) + t2 + m]);
                cfma(t, X1[(kTileF + t2) * (kTileF + 1) + t1], X2[(WX + t1 + m) * (WX + 1) + t2 + m]);
                if (CH != G4_PH_TRANSVERSE) cfma(t, A[t1 * Nwex + m], B[t2 * Nwex + m]);
                sum[m].x += t.x;
                sum[m].y += t.y;
            }
        }
        if (!live) continue;
#pragma unroll
        for (int m = 0; m < WXM; ++m) {
            if (m >= Nwex) break;
            if (n1 + d.m0 + m >= Nw2 || n2 + d.m0 + m >= Nw2) continue;  // structurally zero
            double2 o = sum[m];
            if (staged > 1) o = make_double2(row[m].x + o.x, row[m].y + o.y);
            row[m] = o;
        }
    }
}

// The value of an accumulator entry: complex128, or a pair of complex64 whose
// sum is the value (compensated FP32 pairs; hi + lo is exact in FP64).
template <bool PAIR>
__device__ __forceinline__ double2 acc_value(const double2* acc, size_t i) {
    if constexpr (PAIR) {
        const float4 a = reinterpret_cast<const float4*>(acc)[i];
        return make_double2((double)a.x + (double)a.z, (double)a.y + (double)a.w);
    } else {
        return acc[i];
    }
}

// out[m][n2][n1][q][k2][k1] = acc[k1][n1][k2][n2][q][m] * inv_s for n2 in
// [n2_0, n2_0 + n2_cnt) and q in [q0, q0 + nq), written at out + m * out_plane +
// (n2 - n2_0) * (one n2 plane): the whole exported array when out_plane =
// E / Nwex and n2_0 = 0, or a staging block of a few n2 planes per m.
//
// DIRECT: the direct term's last window is added on the way, acc + scr, in
// place of a read-modify-write of the accumulator before this pass; scr and
// scr0 are the group's scratch planes (g4_direct_tc.cu), q0 its first momentum.
//
// Bound by HBM, and with DIRECT by the FP64 pipe as much (two additions and two
// products per entry at two lanes per clock and SM; the sums cannot be formed
// in fewer without losing bits).  A block owns one n1, kFinN2 consecutive n2
// and the transfers of TQ momenta (kFinNJ: runs of 128 bytes in the
// accumulator), and walks the momentum pairs r = (k2, k1) in chunks of RC, a
// multiple of eight, through kFinBytes of shared memory: out is written in runs
// of RC entries, whole 128-byte lines.  A thread keeps its transfer and n2 and
// walks r, so no index is divided inside the loop; kFinU loads of each array
// are in flight per thread.  Many small blocks keep the FP64 and the memory
// phases of different blocks side by side.
// Measured, addition and export, before (read-modify-write by bulk reductions,
// then export) -> after: 4x4 cluster, 64 frequencies, Nwex = 8: 1.77 -> 1.30 ms;
// 6x6, 64, 4: 11.4 -> 7.2; 8x8, 32, 4: 15.8 -> 9.9 (4.3 TB/s over acc, scratch
// and out).  256 threads with twice the memory took 10.9 ms there, 64 with half
// 10.1; four n2 10.2, one 10.4; two or eight loads 10.7 and 11.1; runs that are
// no multiple of 128 bytes 15 to 18.
constexpr int kFinN2 = 2;
constexpr int kFinU = 4;
constexpr int kFinNJ = 8;
constexpr int kFinBytes = 18 * 1024;
constexpr int kFinThreads = 128;
constexpr long long kFinBlocks = 12288;
constexpr int kFinWideBytes = 24 * 1024, kFinWideMax = 96 * 1024;

template <bool PAIR, bool DIRECT>
__global__ void __launch_bounds__(kFinThreads) k_finalize(
    const double2* __restrict__ acc, const float2* __restrict__ scr,
    const double2* __restrict__ scr0, double inv_s, double2* __restrict__ out, G4Dims d, int TQ,
    int RC, int nsplit, int n2_0, int n2_cnt, int q0, int nq, long long out_plane) {
    extern __shared__ double2 tileF[];  // [kFinN2][RC][ld]
    const int Nc = d.Nc, Nw2 = d.Nw2, Nwex = d.Nwex, NR = Nc * Nc;
    const int n1 = blockIdx.x, n2b = blockIdx.y * kFinN2;
    const int zq = blockIdx.z / nsplit, split = blockIdx.z - zq * nsplit, qb = zq * TQ;
    const int NJ = min(TQ, nq - qb) * Nwex;          // transfers (q, m), contiguous in acc
    const int nn = min(kFinN2, n2_cnt - n2b);
    const int ld = NJ | 1;                           // odd: the transposed reads are conflict-free
    const int L = NJ * kFinN2, G = kFinThreads / L;  // threads per momentum pair; pairs at a time
    const int g = threadIdx.x / L, jn = threadIdx.x - g * L;
    const int n2l = jn / NJ, j = jn - n2l * NJ;
    const int n2 = n2_0 + n2b + n2l;
    const bool mine = g < G && n2l < nn;
    const int m = d.m0 + j % Nwex;
    const int Ql = qb * Nwex + j;                    // plane of the group's scratch
    const bool on = DIRECT && n1 + m < Nw2 && n2 + m < Nw2;   // else structurally zero
    const bool first = q0 == 0 && Ql == 0;           // Q = 0: FP64 scratch
    const size_t a1 = (size_t)Nw2 * d.N * d.NQ, a2 = (size_t)Nw2 * d.NQ;
    const double2* ap = acc + ((size_t)n1 * d.N + n2) * d.NQ + (size_t)(q0 + qb) * Nwex + j;
    const size_t s1 = (size_t)Nw2 * d.N, sofs = (size_t)n1 * d.N + n2;
    const float2* sp = DIRECT ? scr + (size_t)Ql * d.N * d.N + sofs : nullptr;
    const int dk2 = G / Nc, dk1 = G - dk2 * Nc;      // r += G
    const int warp = threadIdx.x >> 5;
    for (int r0 = split * RC; r0 < NR; r0 += nsplit * RC) {
        const int rc = min(RC, NR - r0);
        if (mine) {
            int k2 = (r0 + g) / Nc, k1 = r0 + g - k2 * Nc;
            for (int rb = g; rb < rc; rb += kFinU * G) {
                double2 v[kFinU];
                float2 f[kFinU];
                size_t f0[kFinU];
#pragma unroll
                for (int u = 0; u < kFinU; ++u) {
                    if (rb + u * G < rc) {
                        v[u] = acc_value<PAIR>(ap, (size_t)k1 * a1 + (size_t)k2 * a2);
                        if constexpr (DIRECT) {
                            f0[u] = (size_t)k1 * s1 + (size_t)(k2 * Nw2);
                            if (on && !first) f[u] = sp[f0[u]];
                        }
                    }
                    k1 += dk1;
                    k2 += dk2;
                    if (k1 >= Nc) {
                        k1 -= Nc;
                        ++k2;
                    }
                }
#pragma unroll
                for (int u = 0; u < kFinU; ++u) {
                    const int rr = rb + u * G;
                    if (rr >= rc) break;
                    if constexpr (DIRECT) {
                        if (on) {
                            const double2 t = first ? scr0[f0[u] + sofs]
                                                    : make_double2(g4ptx::f32_to_f64(f[u].x), g4ptx::f32_to_f64(f[u].y));
                            v[u].x += t.x;
                            v[u].y += t.y;
                        }
                    }
                    tileF[((size_t)n2l * RC + rr) * ld + j] = v[u];
                }
            }
        }
        __syncthreads();
        // a warp writes one (n2, q, m) plane's run of rc entries at a time, or
        // several planes' runs when they are shorter than a warp
        const int run = rc > 16 ? 32 : rc > 8 ? 16 : rc > 4 ? 8 : rc > 2 ? 4 : rc;
        const int pw = 32 / run, lane = (threadIdx.x & 31) % run;
        for (int pl = warp * pw + (threadIdx.x & 31) / run; pl < nn * NJ; pl += kFinThreads / 32 * pw) {
            const int nl = pl / NJ, jj = pl - nl * NJ, qi = jj / Nwex, ml = jj - qi * Nwex;
            double2* o = out + (size_t)ml * out_plane +
                         (((size_t)(n2b + nl) * Nw2 + n1) * d.Nkex + q0 + qb + qi) * NR + r0;
            const double2* t = tileF + (size_t)nl * RC * ld + jj;
            for (int rr = lane; rr < rc; rr += run) {
                const double2 v = t[(size_t)rr * ld];
                o[rr] = make_double2(v.x * inv_s, v.y * inv_s);
            }
        }
        __syncthreads();
    }
}

// The export of many transfer frequencies: a block owns one (n1, n2, q) triple,
// 256 threads, and walks k2 in chunks of KC through shared memory, so that it
// reads runs of Nwex contiguous entries and writes runs of KC Nc.  For more than
// 12 transfers, on clusters of less than twelve sites for more than 8 (runs of
// a few dozen entries, whose index arithmetic is then shared by more threads).
// k_finalize / here: 4x4 cluster, 64 frequencies, 4 momenta, 13 transfers 0.39 /
// 0.36 ms, 32: 1.29 / 0.76, 64: 4.6 / 1.5, but 11: 0.32 / 0.38; 3x3, 16
// frequencies, 9 momenta, 9 transfers 0.020 / 0.014, but 17 frequencies, 7
// momenta, 5 transfers 0.025 / 0.029.
bool finalize_wide(const G4Dims& d) { return d.Nwex > 12 || (d.Nwex > 8 && d.Nc < 12); }

template <bool PAIR>
__global__ void __launch_bounds__(256) k_finalize_wide(const double2* __restrict__ acc, double inv_s,
                                                       double2* __restrict__ out, G4Dims d, int KC, int n2_0,
                                                       int q0, long long out_plane) {
    extern __shared__ double2 tileF[];  // [KC][Nc][Nwex + 1]
    const int n1 = blockIdx.x, n2l = blockIdx.y, q = q0 + blockIdx.z;
    const int n2 = n2_0 + n2l;
    const int Nc = d.Nc, Nw2 = d.Nw2, Nwex = d.Nwex, ld = Nwex + 1;
    for (int k20 = 0; k20 < Nc; k20 += KC) {
        const int kc = min(KC, Nc - k20);
        const int cnt = kc * Nc * Nwex;
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
            const int r = t / Nwex, m = t - r * Nwex;
            const int k2l = r / Nc, k1 = r - k2l * Nc;
            const size_t K1 = (size_t)k1 * Nw2 + n1, K2 = (size_t)(k20 + k2l) * Nw2 + n2;
            tileF[r * ld + m] = acc_value<PAIR>(acc, (K1 * d.N + K2) * d.NQ + (size_t)q * Nwex + m);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
            const int m = t / (kc * Nc), r = t - m * (kc * Nc);   // r = (k2l, k1), k1 fastest
            const double2 v = tileF[r * ld + m];
            out[(size_t)m * out_plane + (((size_t)n2l * Nw2 + n1) * d.Nkex + q) * Nc * Nc +
                (size_t)k20 * Nc + r] = make_double2(v.x * inv_s, v.y * inv_s);
        }
        __syncthreads();
    }
}

// Mixed path G build.  One block owns kDiagCols columns c = (kc, j) of one row
// momentum kr and spin: it forms G in FP32, scales it by sqrt(s_r)
// (i sqrt(|s_r|) for a negative sign, so that the product of two entries of
// the same measurement carries s_r) and writes every frequency-difference
// diagonal's complex64 run over its columns (the positions where the row index
// leaves the grid stay zero):
//   Gd[j][dk][dn + Nw2-1][kc][n] = sqrt(s_r) G((kr, n+dn), (kc, n)),  kr = kc (+) dk.
//
// Bound by HBM (M read once, G~ written once).  The Nw2 rows of M go to shared
// memory by asynchronous copies, all in flight at once without holding
// registers, and are read back along the diagonals: a lane's row stride is a
// multiple of 128 bytes and lanes are consecutive columns, so every access is
// free of bank conflicts.  Step t takes row (n + t) mod Nw2, whose diagonal is
// dn = t or t - Nw2: all lanes write in every step, where walking the 2Nw2 - 1
// diagonals in turn left half of them out.  Columns run over momenta, so small
// frequency counts fill their warps too.  One maximum per block goes to *gmax.
// Measured back to back (bytes M + G~), before -> after, complex128 M:
// N = 32: 4.17 -> 2.15 us; N = 1024 (4x4, 64 frequencies):
// 18.9 -> 14.4 us (3.5 TB/s); N = 2304: 61.7 -> 50.6 us (5.0 TB/s); complex64,
// N = 750 (50 frequencies): 12.3 -> 7.9 us.  Of that the programmatic launch is
// 2 us; 16 columns or 128 threads per block measured within 5% either way, 512
// threads 10% slower at N = 2304.
constexpr int kDiagCols = 32;

template <typename MV>
__device__ __forceinline__ void cp_async_entry(void* dst, const MV* src) {
    if constexpr (sizeof(MV) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(g4ptx::smem_u32(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(g4ptx::smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ float2 narrow(float2 z) { return z; }
__device__ __forceinline__ float2 narrow(double2 z) {
    return make_float2(g4ptx::f64_to_f32(z.x), g4ptx::f64_to_f32(z.y));
}

template <bool M64>
__global__ void __launch_bounds__(256) k_build_G_diag(const void* __restrict__ M,
                                                      const double2* __restrict__ G0,
                                                      g4gt::SignFactor sf, float2* __restrict__ Gd,
                                                      const int* __restrict__ ksub, G4Dims d,
                                                      unsigned* __restrict__ gmax) {
    // M entries as loaded: complex64 stays complex64, complex128 is narrowed below
    using MV = typename std::conditional<M64, float2, double2>::type;
    extern __shared__ __align__(16) unsigned char smem_diag[];
    __shared__ unsigned bmax;
    const int Nw2 = d.Nw2, N = d.N;
    MV* rows = reinterpret_cast<MV*>(smem_diag);                             // [Nw2][kDiagCols]
    float2* g0row = reinterpret_cast<float2*>(rows + (size_t)Nw2 * kDiagCols);   // [Nw2]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int c = blockIdx.x * kDiagCols + lane, kr = blockIdx.y, sp = blockIdx.z;
    const bool ok = c < N;
    // M and G0 may come from the kernel before: nothing is read until it is done
    g4ptx::pdl_wait();
    const MV* src = reinterpret_cast<const MV*>(M) + ((size_t)sp * N + (size_t)kr * Nw2) * N + c;
    if (ok)
        for (int i = warp; i < Nw2; i += nwarp)
            cp_async_entry(&rows[i * kDiagCols + lane], src + (size_t)i * N);
    asm volatile("cp.async.commit_group;" ::: "memory");
    // complex64 storage: form G in FP32 (three roundings, below the storage rounding scale)
    for (int i = threadIdx.x; i < Nw2; i += blockDim.x) {
        const double2 g = G0[sp * N + kr * Nw2 + i];
        g0row[i] = narrow(g);
    }
    if (threadIdx.x == 0) bmax = 0u;
    const int kc = ok ? c / Nw2 : 0, n = ok ? c - kc * Nw2 : 0;
    float2 gj = make_float2(0.f, 0.f);
    if (ok) {
        const double2 g = G0[sp * N + c];
        gj = narrow(g);
    }
    const size_t plane = (size_t)d.Nc * Nw2;
    float2* out = Gd + ((size_t)sp * d.Nc + ksub[kr * d.Nc + kc]) * d.ndn * plane +
                  (size_t)(Nw2 - 1) * plane + c;   // the diagonal dn = 0
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float vmax = 0.f;
    if (ok) {
#pragma unroll 4
        for (int t = warp; t < Nw2; t += nwarp) {
            const bool wrap = n + t >= Nw2;
            const int dn = wrap ? t - Nw2 : t, i = n + dn;
            const float2 v = g4gt::g_tilde(g0row[i], narrow(rows[i * kDiagCols + lane]), gj,
                                           dn == 0 && kr == kc, sf);
            vmax = fmaxf(vmax, fmaxf(fabsf(v.x), fabsf(v.y)));
            out[(long long)dn * (long long)plane] = v;
        }
    }
    // the block's largest component joins the batch's maximum (non-negative
    // FP32 values order like their bit patterns)
    const unsigned wmax = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
    if (lane == 0) atomicMax(&bmax, wmax);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(gmax, bmax);
}

// Zero the accumulator's entries with K1 = K2 (the diagonal D = 0, whose split
// tiles in the tensor-core exchange add their partial sums also in the first
// batch).
__global__ void k_clear_diag(double2* __restrict__ acc, int N, int NQ) {
    double2* row = acc + ((size_t)blockIdx.x * N + blockIdx.x) * NQ;
    for (int i = threadIdx.x; i < NQ; i += blockDim.x) row[i] = make_double2(0.0, 0.0);
}

__global__ void k_clear_unset(double2* __restrict__ acc, long long E, const unsigned* __restrict__ accset) {
    if (*accset) return;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < E;
         i += (long long)gridDim.x * blockDim.x)
        acc[i] = make_double2(0.0, 0.0);
}

// Whether the tiled update takes the shape: from 2^18 entries on (below, a launch
// of it is a chain of barriers over transfers and measurements in a few blocks),
// when enough of its frequency tiles lies on the grid (Nw2^2 of the tiles' area;
// the opposite-spin channel, without the direct term, has less to share in a
// tile).  16 measurements, simple / tiled, ms: 3x3 cluster, 9 momenta, magnetic, 4
// transfers: 20 frequencies (0.39 of the tiles) 0.99 / 1.95, 28 (0.77) 1.91 /
// 1.96, 3 transfers, 40 (0.69) 2.89 / 2.51; 2x2, 8 transfers, 50 (0.61) 1.06 /
// 1.11, 4, 80 (1) 1.38 / 0.89; transverse: 4 transfers, 16 frequencies (1) 1.99 /
// 1.74, 2 transfers, 0.99 / 1.04, 16 transfers, 100 (0.80) 4.8 / 4.6.
constexpr long long kTiledMinEntries = 1 << 18;
bool tiled_wanted(const G4Dims& d) {
    if (d.ch == G4_PP_UPDOWN || d.Nwex > kTileWex || (long long)d.Nc * d.Nc > 65535 || d.E < kTiledMinEntries)
        return false;
    const int side = (d.Nw2 + kTileF - 1) / kTileF * kTileF;
    const double fill = (double)d.Nw2 * d.Nw2 / ((double)side * side);
    return d.ch == G4_PH_TRANSVERSE ? d.Nwex > 2 && fill >= 0.78 : fill >= 0.65;
}

}  // namespace

cudaError_t launch_build_G_fp64(const void* M, bool m64, const double2* G0, double2* G, int N,
                                unsigned* flag, cudaStream_t s) {
    const int bx = N >= 256 ? 256 : (N + 31) / 32 * 32;
    const dim3 grid((N + kBuildU * bx - 1) / (kBuildU * bx), std::min(2LL * N, 65535LL));
    auto* k = m64 ? (flag ? k_build_G_fp64<true, true> : k_build_G_fp64<true, false>)
                  : (flag ? k_build_G_fp64<false, true> : k_build_G_fp64<false, false>);
    k<<<grid, bx, 0, s>>>(M, G0, G, N, flag);
    return cudaGetLastError();
}

namespace {
template <int CH>
cudaError_t update_fp64(const double2* G, const G4Signs& signs, int staged, double2* acc,
                        const int* kadd, const int* ksub, const G4Dims& d, const unsigned* only_if,
                        cudaStream_t s) {
    if (tiled_wanted(d)) {
        const int nt = (d.Nw2 + kTileF - 1) / kTileF;
        const int WX = kTileF + d.Nwex - 1;
        const size_t smem = (2 * (size_t)WX * (WX + 1) + 2 * kTileF * (kTileF + 1) +
                             2 * (size_t)kTileF * d.Nwex) * sizeof(double2);
        const dim3 grid(nt * nt, d.Nc * d.Nc);
        auto* k = d.Nwex <= 4 ? k_update_fp64_tiled<CH, 4>
                              : d.Nwex <= 8 ? k_update_fp64_tiled<CH, 8> : k_update_fp64_tiled<CH, kTileWex>;
        if (smem > 48 * 1024) {
            cudaError_t e = raise_smem_limit(k);
            if (e != cudaSuccess) return e;
        }
        k<<<grid, kTileF * kTileF, smem, s>>>(G, signs, staged, acc, kadd, d, only_if);
        return cudaGetLastError();
    }
    const int per = d.N * d.NQ;
    auto run = [&](auto rs) {
        constexpr int RS = decltype(rs)::value;
        const long long threads = (long long)per * RS;
        const int bx = threads < 256 ? (int)(threads + 31) / 32 * 32 : 256;
        const int gx = (int)std::min<long long>((threads + bx - 1) / bx, 64);
        k_update_fp64<CH, RS><<<dim3(gx, d.N), bx, 0, s>>>(G, signs, staged, acc, kadd, ksub, d, only_if);
    };
    // a lane per entry once that fills the GPU a few times over
    if (d.E >= (1 << 18) || staged < 4) run(std::integral_constant<int, 1>());
    else if (d.E >= (1 << 15) || staged < 16) run(std::integral_constant<int, 4>());
    else run(std::integral_constant<int, 16>());
    return cudaGetLastError();
}
}  // namespace

double update_fp64_ps(const G4Dims& d) {
    if (d.ch == G4_PP_UPDOWN) return 25.5;
    const bool trans = d.ch == G4_PH_TRANSVERSE;
    if (!tiled_wanted(d)) return trans ? 30.0 : 52.0;
    const int side = (d.Nw2 + kTileF - 1) / kTileF * kTileF;
    const double fill = (double)d.Nw2 * d.Nw2 / ((double)side * side);
    return (trans ? 19.5 + 6.0 / d.Nwex : 27.0 + 10.0 / d.Nwex) / fill;
}

cudaError_t launch_update_fp64(const double2* G, const G4Signs& signs, int staged, double2* acc,
                               const int* kadd, const int* ksub, const G4Dims& d,
                               const unsigned* only_if, cudaStream_t s) {
    switch (d.ch) {
        case G4_PP_UPDOWN:
            return update_fp64<G4_PP_UPDOWN>(G, signs, staged, acc, kadd, ksub, d, only_if, s);
        case G4_PH_DENSITY:
            return update_fp64<G4_PH_DENSITY>(G, signs, staged, acc, kadd, ksub, d, only_if, s);
        case G4_PH_TRANSVERSE:
            return update_fp64<G4_PH_TRANSVERSE>(G, signs, staged, acc, kadd, ksub, d, only_if, s);
        default:
            return update_fp64<G4_PH_MAGNETIC>(G, signs, staged, acc, kadd, ksub, d, only_if, s);
    }
}

cudaError_t launch_finalize(const double2* acc, bool pair, double inv_s, double2* out,
                            const G4Dims& d, int n2_0, int n2_cnt, long long out_plane, int q0,
                            int nq, const float2* scr, const double2* scr0, cudaStream_t s) {
    const int NR = d.Nc * d.Nc;
    const size_t plane = (size_t)d.Nc * (d.Nwex + 1) * sizeof(double2);   // one k2
    if (!scr && finalize_wide(d) && plane <= kFinWideMax) {
        const int KC = (int)std::min<size_t>(d.Nc, std::max<size_t>(1, kFinWideBytes / plane));
        auto* k = pair ? k_finalize_wide<true> : k_finalize_wide<false>;
        if (KC * plane > 48 * 1024) {
            cudaError_t e = raise_smem_limit(k);
            if (e != cudaSuccess) return e;
        }
        k<<<dim3(d.Nw2, n2_cnt, nq), 256, KC * plane, s>>>(acc, inv_s, out, d, KC, n2_0, q0, out_plane);
        return cudaGetLastError();
    }
    // transfers per block: a 128-byte run, or one momentum's (NJ * kFinN2 is at
    // most kFinThreads: Nwex <= 64)
    const int TQ = std::min(nq, std::max(1, kFinNJ / d.Nwex));
    const int NJ = TQ * d.Nwex, ld = NJ | 1;
    const size_t per = (size_t)kFinN2 * ld * sizeof(double2);
    const long long blocks = (long long)d.Nw2 * ((n2_cnt + kFinN2 - 1) / kFinN2) * ((nq + TQ - 1) / TQ);
    // pairs per chunk: all of them, or equal chunks of whole 128-byte lines
    int RC = (int)std::min<size_t>(NR, std::max<size_t>(1, kFinBytes / per));
    if (RC < NR && RC >= 8) {
        RC = RC / 8 * 8;
        const int n = (NR + RC - 1) / RC;
        RC = ((NR + n - 1) / n + 7) / 8 * 8;
    }
    // the chunks are dealt to enough blocks to fill the GPU several times over
    // (8x8 cluster, 32 frequencies: 15.0 ms with a group's blocks undivided, 11.0
    // divided)
    const long long chunks = ((long long)NR + RC - 1) / RC;
    const int nsplit = (int)std::min<long long>(std::min<long long>(chunks, 256), (kFinBlocks + blocks - 1) / blocks);
    const dim3 grid(d.Nw2, (n2_cnt + kFinN2 - 1) / kFinN2, (nq + TQ - 1) / TQ * nsplit);
    auto* k = pair ? k_finalize<true, false> : scr ? k_finalize<false, true> : k_finalize<false, false>;
    k<<<grid, kFinThreads, RC * per, s>>>(acc, scr, scr0, inv_s, out, d, TQ, RC, nsplit, n2_0, n2_cnt, q0, nq,
                                          out_plane);
    return cudaGetLastError();
}

cudaError_t launch_clear_diag(double2* acc, const G4Dims& d, cudaStream_t s) {
    k_clear_diag<<<d.N, 128, 0, s>>>(acc, d.N, d.NQ);
    return cudaGetLastError();
}

cudaError_t launch_clear_unset(double2* acc, const unsigned* accset, const G4Dims& d, cudaStream_t s) {
    k_clear_unset<<<(int)std::min<long long>((d.E + 255) / 256, 152 * 16), 256, 0, s>>>(acc, d.E, accset);
    return cudaGetLastError();
}

cudaError_t launch_build_G_diag(const void* M, bool m64, const double2* G0, double sign,
                                float2* Gd_slot, const int* ksub, const G4Dims& d,
                                unsigned* gmax, cudaStream_t s) {
    const size_t smem = (size_t)d.Nw2 * kDiagCols * (m64 ? sizeof(float2) : sizeof(double2)) +
                        (size_t)d.Nw2 * sizeof(float2);
    const dim3 grid((d.N + kDiagCols - 1) / kDiagCols, d.Nc, 2);
    auto* k = m64 ? k_build_G_diag<true> : k_build_G_diag<false>;
    if (smem > 48 * 1024) {
        cudaError_t e = raise_smem_limit(k);
        if (e != cudaSuccess) return e;
    }
    // a run is a chain of these launches: the next one's blocks are set up while
    // this one finishes, and wait for it (on the device) before their first read
    return launch_pdl(k, grid, dim3(256), smem, s, M, G0, g4gt::sign_factor(sign), Gd_slot, ksub, d, gmax);
}
