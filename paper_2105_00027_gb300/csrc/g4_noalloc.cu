// Allocation-free entry point: one measurement's plain FP64 update of a
// caller-owned accumulator, with the intermediate G kept in a fixed,
// file-scope device array instead of memory from cudaMalloc.
//
// Who needs it: callers that cannot allocate device memory at the point of
// the update -- for example code whose device memory is owned by another
// allocator that has already reserved the GPU (a framework's caching
// allocator), or a measurement loop that must not pay the implicit device
// synchronisation of cudaMalloc/cudaFree.  Everything this path needs beyond
// the caller's inputs and output lives in g4_noalloc_G below.
//
// The array is shared by every call in the process: calls whose work overlaps
// on the GPU (different streams, or different host threads) race on it.  It
// keeps the last call's contents; each call overwrites all of it that it
// reads, so nothing needs clearing between calls.
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "g4_internal.h"

namespace {

constexpr int kMaxN = G4_NOALLOC_MAX_N;

// Scratch for G of both spins: 2 * 256 * 256 complex128 = 2 MiB per device,
// held by every GPU that loads the library until the process exits.
static __device__ __align__(256) double2 g4_noalloc_G[2 * kMaxN * kMaxN];

// Device address of the array, looked up once per device and context (host
// code must not use the symbol itself: on the host it is only a stand-in).
// The address belongs to the context that was current at the lookup; after
// cudaDeviceReset the device gets a new primary context, so the identifier of
// the current context is kept beside the address and a change triggers a new
// lookup.
std::mutex g_mu;
double2* g_ptr[256] = {};
unsigned long long g_ctx[256] = {};

__device__ __forceinline__ double2 na_cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__global__ void k_na_build(const double2* __restrict__ M, const double2* __restrict__ G0,
                           double2* __restrict__ G, int N) {
    const size_t NN = (size_t)N * N;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < 2 * NN;
         e += (size_t)gridDim.x * blockDim.x) {
        const int sp = (int)(e / NN);
        const size_t ij = e - (size_t)sp * NN;
        const int i = (int)(ij / N), j = (int)(ij - (size_t)i * N);
        const double2 gi = G0[sp * N + i], gj = G0[sp * N + j];
        double2 v = na_cmul(na_cmul(gi, M[e]), gj);
        v.x = -v.x;
        v.y = -v.y;
        if (i == j) {
            v.x += gi.x;
            v.y += gi.y;
        }
        G[e] = v;
    }
}

// acc[m][n2][n1][q][k2][k1] += sign * (a b - exchange).  A block takes gp
// consecutive (n1, q) of one n2 (blockIdx.y), its threads the gp Nc^2 pairs
// (k2, k1) of each, and walks the transfers m in steps of kNaM: a (with the
// sign) and b of the step are formed once into shared memory, G(K2, K1) is read
// once per entry, the kNaM accumulator entries and G(K1+Q, K2+Q) are read
// together.  Bound by the FP64 pipe (two lanes per clock and SM): fourteen
// operations per entry, and no index division or weighted sum per entry (one
// thread per entry with both took 211 us for N = 256 and 64 transfers; this
// 110).  The contribution is summed before it meets the accumulator: with the
// accumulator inside the chain of fused multiply-adds, two operations fewer
// (95 us), the error against 64 bits grew by half.
//
// Where the (n1, q) groups and n2 are too few blocks to fill the GPU, the
// transfer steps (blockIdx.z % nm) and then the pairs (blockIdx.z / nm) are
// dealt to several; each forms its own a and b.  Ten calls, one thread per entry
// / groups alone / dealt: 16x8 cluster, N = 256, one transfer: 0.16 / 1.17 /
// 0.16 ms; 8x8, 4 frequencies, 4 transfers: 0.24 / 0.80 / 0.22; 1x1, 128
// frequencies, 64 transfers: 0.60 / 0.85 / 0.46.
constexpr int kNaM = 4;
constexpr int kNaThreads = 256;
constexpr int kNaBlocks = 152 * 8;   // blocks that fill the GPU

__device__ __forceinline__ void na_cfma(double2& t, double2 a, double2 b) {
    t.x = fma(a.x, b.x, t.x);
    t.y = fma(a.x, b.y, t.y);
    t.x = fma(-a.y, b.y, t.x);
    t.y = fma(a.y, b.x, t.y);
}

template <bool DEAL>
__global__ void __launch_bounds__(kNaThreads, 3) k_na_update(const double2* __restrict__ G, double sign,
                                                          double2* __restrict__ acc, int Nc, int Lx,
                                                          int Nw2, int Nwex, int Nkex, int gp, int nm) {
    __shared__ double2 sa[kNaM * kNaThreads], sb[kNaM * kNaThreads];   // [m][group][k]
    const int N = Nc * Nw2, Ly = Nc / Lx, N2 = Nc * Nc;
    const size_t NN = (size_t)N * N;
    const int n2 = blockIdx.y, g0 = blockIdx.x * gp, ng = min(gp, Nw2 * Nkex - g0);
    const size_t plane = (size_t)Nw2 * Nkex * N2;   // entries of one (m, n2)
    auto add = [&](int k, int q) {
        int x = k % Lx + q % Lx, y = k / Lx + q / Lx;
        x -= x >= Lx ? Lx : 0;
        y -= y >= Ly ? Ly : 0;
        return x + Lx * y;
    };
    const int zm = DEAL ? blockIdx.z % nm : 0, mstep = DEAL ? nm * kNaM : kNaM;
    const int t0 = DEAL ? blockIdx.z / nm * blockDim.x + threadIdx.x : threadIdx.x;
    const int tstep = DEAL ? gridDim.z / nm * blockDim.x : blockDim.x;
    for (int m0 = zm * kNaM; m0 < Nwex; m0 += mstep) {
        __syncthreads();
        for (int t = threadIdx.x; t < ng * Nc; t += blockDim.x) {
            const int g = t / Nc, k = t - g * Nc;
            const int n1 = (g0 + g) / Nkex, q = (g0 + g) - n1 * Nkex;
            const int kq = add(k, q);
#pragma unroll
            for (int u = 0; u < kNaM; ++u) {
                const int m = m0 + u;
                double2 a = make_double2(0.0, 0.0), b = a;
                if (m < Nwex && n1 + m < Nw2) {
                    const size_t e = (size_t)(kq * Nw2 + n1 + m) * N + k * Nw2 + n1;
                    const double2 x = G[e], y = G[NN + e];
                    a = make_double2(sign * (x.x - y.x), sign * (x.y - y.y));
                }
                if (m < Nwex && n2 + m < Nw2) {
                    const size_t e = (size_t)(k * Nw2 + n2) * N + kq * Nw2 + n2 + m;
                    const double2 x = G[e], y = G[NN + e];
                    b = make_double2(x.x - y.x, x.y - y.y);
                }
                sa[u * kNaThreads + t] = a;
                sb[u * kNaThreads + t] = b;
            }
        }
        __syncthreads();
        for (int t = DEAL ? t0 : threadIdx.x; t < ng * N2; t += DEAL ? tstep : blockDim.x) {
            const int g = t / N2, r = t - g * N2, k2 = r / Nc, k1 = r - k2 * Nc;
            const int n1 = (g0 + g) / Nkex, q = (g0 + g) - n1 * Nkex;
            const int lim = min(Nwex, Nw2 - max(n1, n2)) - m0;   // transfers on the grid
            if (lim <= 0) continue;
            const size_t e1 = (size_t)(k2 * Nw2 + n2) * N + k1 * Nw2 + n1;
            const size_t e2 = (size_t)(add(k1, q) * Nw2 + n1 + m0) * N + add(k2, q) * Nw2 + n2 + m0;
            double2* o = acc + (size_t)m0 * Nw2 * plane + (size_t)n2 * plane + (size_t)g0 * N2 + t;
            double2 x1[2], x2[kNaM][2], s[kNaM];
#pragma unroll
            for (int sp = 0; sp < 2; ++sp) {
                x1[sp] = G[sp * NN + e1];
                x1[sp] = make_double2(-sign * x1[sp].x, -sign * x1[sp].y);
            }
#pragma unroll
            for (int u = 0; u < kNaM; ++u)
                if (u < lim) {
                    s[u] = o[(size_t)u * Nw2 * plane];
#pragma unroll
                    for (int sp = 0; sp < 2; ++sp) x2[u][sp] = G[sp * NN + e2 + (size_t)u * (N + 1)];
                }
#pragma unroll
            for (int u = 0; u < kNaM; ++u)
                if (u < lim) {
                    double2 v = na_cmul(x1[0], x2[u][0]);
                    na_cfma(v, x1[1], x2[u][1]);
                    na_cfma(v, sa[u * kNaThreads + g * Nc + k1], sb[u * kNaThreads + g * Nc + k2]);
                    o[(size_t)u * Nw2 * plane] = make_double2(s[u].x + v.x, s[u].y + v.y);
                }
        }
    }
}

// Errors are reported like those of g4_create: message via g4_last_error(NULL).
g4_status na_fail(g4_status st, const std::string& msg) { return g4_fail(nullptr, st, msg); }

// Identifier of the current context (driver cuCtxGetId, reached through the
// runtime's entry-point query so that nothing links against libcuda), or 0
// when it cannot be read.
unsigned long long current_ctx_id() {
    static PFN_cuCtxGetId_v12000 get_id = nullptr;
    static PFN_cuCtxGetCurrent_v4000 get_cur = nullptr;
    static bool looked = false;
    if (!looked) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = (PFN_cuCtxGetId_v12000)p;
        p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 4000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_cur = (PFN_cuCtxGetCurrent_v4000)p;
        looked = true;
    }
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_id || !get_cur || get_cur(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

// Set-up for the current device: find the device address of the scratch
// array.  Runs inside the first call on each device (and again when that
// device's context has been replaced, e.g. after cudaDeviceReset).
g4_status na_scratch(double2** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_fail(G4_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= 256) return na_fail(G4_ERR_CUDA, "device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_mu);
    // the context identifier is read after the lookup on the first call (the
    // lookup is what brings the runtime's context up), before it afterwards
    if (!g_ptr[dev] || current_ctx_id() != g_ctx[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g4_noalloc_G);
        if (e != cudaSuccess || !p)
            return na_fail(G4_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        g_ptr[dev] = (double2*)p;
        g_ctx[dev] = current_ctx_id();
    }
    *out = g_ptr[dev];
    return G4_OK;
}

}  // namespace

extern "C" g4_status g4_update_noalloc(int Nc, int lx, int Nw, int Nwex, int Nkex, const void* M,
                                       const void* G0, double sign, void* acc, void* stream) {
    if (!M || !G0 || !acc) return na_fail(G4_ERR_INVALID, "M, G0 or acc is NULL");
    // the same limits as g4_create
    if (Nc < 1 || Nc > 256 || Nw < 1 || Nw > 64 || Nwex < 1 || Nwex > 64 || Nkex < 1 || Nkex > Nc)
        return na_fail(G4_ERR_INVALID, "problem sizes out of range");
    int Lx = lx;
    if (Lx == 0) {
        Lx = 1;
        while ((Lx + 1) * (Lx + 1) <= Nc) ++Lx;
        if (Lx * Lx != Nc) return na_fail(G4_ERR_INVALID, "Nc is not square; pass lx");
    }
    if (Lx < 1 || Nc % Lx != 0) return na_fail(G4_ERR_INVALID, "lx does not divide Nc");
    const long long N = (long long)Nc * 2 * Nw;
    if (N > kMaxN)
        return na_fail(G4_ERR_INVALID, "Nc*2*Nw = " + std::to_string(N) +
                                           " exceeds the allocation-free limit of " +
                                           std::to_string(kMaxN));
    double2* G = nullptr;
    g4_status st = na_scratch(&G);
    if (st != G4_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t total = 2 * (size_t)N * N;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_na_build<<<blocks, 256, 0, s>>>((const double2*)M, (const double2*)G0, G, (int)N);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(G4_ERR_CUDA, std::string("build launch: ") + cudaGetErrorString(e));
    // (n1, q) groups per block: as many whole Nc x Nc planes as its threads hold
    const int gp = std::max(1, kNaThreads / (Nc * Nc)), groups = 2 * Nw * Nkex;
    const int bx = (groups + gp - 1) / gp, blocks2 = bx * 2 * Nw;
    const int nm = std::min((Nwex + kNaM - 1) / kNaM, (kNaBlocks + blocks2 - 1) / blocks2);
    const int np = std::min((std::min(gp, groups) * Nc * Nc + kNaThreads - 1) / kNaThreads,
                            (kNaBlocks + blocks2 * nm - 1) / (blocks2 * nm));
    auto* k = nm * np > 1 ? k_na_update<true> : k_na_update<false>;
    k<<<dim3(bx, 2 * Nw, nm * np), kNaThreads, 0, s>>>(G, sign, (double2*)acc, Nc, Lx, 2 * Nw, Nwex, Nkex, gp, nm);
    e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(G4_ERR_CUDA, std::string("update launch: ") + cudaGetErrorString(e));
    return G4_OK;
}
