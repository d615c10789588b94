// Allocation-free solve of one subdomain's local problem (no counterpart in
// the paper; a deployment variant of the local factor + solve kernels).
//
// Some callers cannot allocate device memory at all: code running inside a
// host application that owns every device allocation through its own pool
// (and forbids driver allocations once its time loop runs), plug-ins that may
// only touch the buffers handed to them, or real-time loops where a
// cudaMalloc would stall the device.  mrcm_box_solve_noalloc needs only the
// caller's input and output buffers: its scratch (the slab block inverses,
// the per-cell coefficients and the forward-sweep results) lives in a
// file-scope __device__ array of fixed size, which every GPU that loads the
// library holds until the process exits.
#include <cuda_runtime.h>

#include <mutex>
#include <string>

#include "mrcm_internal.h"
#include "mrcm_sweep64.cuh"

namespace {

constexpr int kNaMaxCells = 4096;
constexpr int kNaMaxBlock = mrcm::kSw64B;
constexpr long long kNaMaxW = 262144;       // doubles of slab block inverses (2 MB)
constexpr long long kNaScratch = kNaMaxW + 5LL * kNaMaxCells;

// Shared scratch of every call on this device: W blocks, then d, t_u, t_v,
// t_s and the sweep vector (kNaMaxCells doubles each).
static __device__ __align__(256) double g_noalloc_scratch[kNaScratch];

struct BoxArgs {
    int sz[3];
    int sa, ua, va, su, b, ns, N;
    double h[3];
    int side_type[6];       // 0 no-flow, 1 Robin, 2 Dirichlet
    int side_off[6];        // offset of each side's faces in g / beta / q
};

__device__ __forceinline__ void box_coords(const BoxArgs& a, int c, int lc[3]) {
    const int sl = c / a.b, r = c - sl * a.b, v = r / a.su;
    lc[a.sa] = sl;
    lc[a.ua] = r - v * a.su;
    lc[a.va] = v;
}

// face index of cell (lc) on side (axis, hi) within that side's list:
// tangential axes t1 < t2, t2 slow
__device__ __forceinline__ int side_face(const BoxArgs& a, int axis, const int lc[3]) {
    const int t1 = axis == 0 ? 1 : 0, t2 = axis == 2 ? 1 : 2;
    return lc[t1] + a.sz[t1] * lc[t2];
}

// Transmissibility of the face between cells of permeability k1 and k2, and the
// Robin and Dirichlet half-cell ones (reciprocals in integers instead of divisions).
__device__ __forceinline__ double t_inner(double ah, double k1, double k2) { return 2.0 * ah * k1 * k2 * mrcm::rcp64(k1 + k2); }
__device__ __forceinline__ double t_robin(double area, double h, double k, double beta) {
    return area * mrcm::rcp64(fma(0.5 * h, mrcm::rcp64(k), beta));
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// One box on a cluster of two CTAs that eliminate its slabs from both ends:
//   CTA 0: S_s = D_s - t W_{s-1} t for s = 0 .. h-1, CTA 1: S_s = D_s - t W_{s+1} t
//   for s = ns-1 .. h+1, then the middle slab S_h with both terms,
// each S_s inverted on register tiles (mrcm_sweep64.cuh); the one right-hand side
// is eliminated along (Y_s = W_s (r_s + t Y_prev)) and the solution runs outwards
// from the middle slab, x_s = Y_s + W_s t x_next.
//
// Bound: the pivot chain and the FP64 unit of one SM (about 64 FP64 warp
// instructions a pivot at b = 50), so a second SM halves it; the two chains meet
// once (cluster barrier).  10 x 10 x 5 cells (500 pivots): 1915 us with a packed
// triangle in shared memory on one CTA (an index division and three FP64
// operations per entry, one FP64 division per thread and pivot), 318 us now.
template <int NTH>
__global__ void __launch_bounds__(NTH)
k_box_solve_noalloc(BoxArgs a, const double* __restrict__ K, const double* __restrict__ f,
                    const double* __restrict__ g, const double* __restrict__ beta, double* __restrict__ p,
                    double* __restrict__ q, double* scratch, int* __restrict__ not_spd) {
    using namespace mrcm;
    __shared__ __align__(16) Sweep64Shared<1> sh;
    __shared__ double z[kNaMaxBlock], tv[kNaMaxBlock], tw[kNaMaxBlock];
    __shared__ double part[NTH];
    __shared__ int other_bad;
    const int N = a.N, b = a.b;
    const int half = (int)(blockIdx.x & 1);
    const int h = (a.ns - 1) / 2;                                   // middle slab (CTA 0's)
    const int c_lo = half ? (h + 1) * b : 0, c_hi = half ? N : (h + 1) * b;
    double* W = scratch;
    double* cd = scratch + kNaMaxW;
    double* cu = cd + kNaMaxCells;
    double* cv = cu + kNaMaxCells;
    double* cs = cv + kNaMaxCells;
    double* y = cs + kNaMaxCells;
    const int nx = a.sz[0], ny = a.sz[1];
    const double area[3] = {a.h[1] * a.h[2], a.h[0] * a.h[2], a.h[0] * a.h[1]};
    const double vol = a.h[0] * a.h[1] * a.h[2];
    double ah[3], ih[3];
    for (int ax = 0; ax < 3; ++ax) { ih[ax] = rcp64(a.h[ax]); ah[ax] = area[ax] * ih[ax]; }
    if (threadIdx.x == 0) { sh.bad = 0; other_bad = 0; }
    // ---- coefficients and right-hand side (kept in y) of this CTA's slabs
    for (int c = c_lo + threadIdx.x; c < c_hi; c += NTH) {
        int lc[3];
        box_coords(a, c, lc);
        const int gc = lc[0] + nx * (lc[1] + ny * lc[2]);
        double d = 0.0, tp[3] = {0.0, 0.0, 0.0}, rhs = f[gc] * vol;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const double ka = K[(long long)ax * N + gc];
            const int stride = ax == 0 ? 1 : ax == 1 ? nx : nx * ny;
#pragma unroll
            for (int hi = 0; hi < 2; ++hi) {
                const bool inside = hi ? lc[ax] + 1 < a.sz[ax] : lc[ax] > 0;
                if (inside) {
                    const double T = t_inner(ah[ax], ka, K[(long long)ax * N + gc + (hi ? stride : -stride)]);
                    d += T;
                    if (hi) tp[ax] = T;
                    continue;
                }
                const int sd = 2 * ax + hi;
                const int fi = a.side_off[sd] + side_face(a, ax, lc);
                if (a.side_type[sd] == 1) {
                    const double TR = t_robin(area[ax], a.h[ax], ka, beta[fi]);
                    d += TR;
                    rhs += TR * g[fi];
                } else if (a.side_type[sd] == 2) {
                    const double TD = 2.0 * ah[ax] * ka;
                    d += TD;
                    rhs += TD * g[fi];
                }
            }
        }
        cd[c] = d;
        cu[c] = tp[a.ua];
        cv[c] = tp[a.va];
        cs[c] = tp[a.sa];
        y[c] = rhs;
    }
    cluster_sync();                                                  // CTA 1 couples to the middle slab's cs
    // the register tile of this thread
    const int nt = (b + kSw64T - 1) / kSw64T;
    int ti, tj;
    sweep64_tile(threadIdx.x, ti, tj);
    const bool own = ti < nt && threadIdx.x + 32 < NTH;             // the last warp forms the pivots
    if (!own) ti = tj = 0;
    const int i0 = ti * kSw64T, j0 = tj * kSw64T;
    double m[kSw64T][kSw64T];
#pragma unroll
    for (int r = 0; r < kSw64T; ++r)
#pragma unroll
        for (int c = 0; c < kSw64T; ++c) m[r][c] = 0.0;
    // sum_k W_s[k][i] z[k], rows i spread over the CTA in P parts of the sum; handed to store(i, sum)
    const int P = NTH / b, per = (b + P - 1) / P;
    auto gemv = [&](int sl, auto store) {
        const double* Ws = W + (long long)sl * b * b;
        const int i = threadIdx.x % b, pt = threadIdx.x / b;
        if (pt < P) {
            double s0 = 0.0, s1 = 0.0;
            const int k1 = min(b, (pt + 1) * per);
            int k = pt * per;
            for (; k + 1 < k1; k += 2) {
                s0 = fma(Ws[(long long)k * b + i], z[k], s0);
                s1 = fma(Ws[(long long)(k + 1) * b + i], z[k + 1], s1);
            }
            if (k < k1) s0 = fma(Ws[(long long)k * b + i], z[k], s0);
            part[threadIdx.x] = s0 + s1;
        }
        __syncthreads();
        if (threadIdx.x < b) {
            double s0 = part[threadIdx.x];
            for (int t = 1; t < P; ++t) s0 += part[t * b + threadIdx.x];
            store(threadIdx.x, s0);
        }
        __syncthreads();
    };
    // S_s = D_s - tv W_prev tv (W_prev in the registers) - tw W_other tw (read back), its inverse,
    // and Y_s = W_s (r_s + tv Y_prev + tw Y_other); prev / other < 0: no such neighbour
    auto eliminate = [&](int sl, int prev, int other) {
        const int base = sl * b;
        __syncthreads();
        for (int i = threadIdx.x; i < b; i += NTH) {
            const double t1 = prev < 0 ? 0.0 : cs[min(prev, sl) * b + i];
            const double t2 = other < 0 ? 0.0 : cs[min(other, sl) * b + i];
            tv[i] = t1;
            tw[i] = t2;
            double zi = y[base + i];
            if (prev >= 0) zi = fma(t1, y[prev * b + i], zi);
            if (other >= 0) zi = fma(t2, y[other * b + i], zi);
            z[i] = zi;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSw64T; ++r) {
            const int i = i0 + r;
#pragma unroll
            for (int c = 0; c < kSw64T; ++c) {
                const int j = j0 + c;
                if (i >= b || j >= b) { m[r][c] = 0.0; continue; }
                const int lo = min(i, j), hi = max(i, j);
                double dij = 0.0;
                if (i == j) dij = cd[base + i];
                if (hi == lo + 1 && hi % a.su > 0) dij = -cu[base + lo];
                if (hi == lo + a.su) dij = -cv[base + lo];
                if (other >= 0) dij = fma(-tw[i] * tw[j], W[(long long)other * b * b + (long long)i * b + j], dij);
                m[r][c] = fma(-tv[i] * tv[j], m[r][c], dij);
            }
        }
        sweep64_invert<1>(m, ti, tj, own, b, sh);
        sweep64_store(m, ti, tj, own, b, W + (long long)sl * b * b);
        __syncthreads();
        gemv(sl, [&](int i, double v) { y[base + i] = v; });
    };
    if (half == 0) {
        for (int sl = 0; sl < h; ++sl) eliminate(sl, sl - 1, -1);
    } else {
        for (int sl = a.ns - 1; sl > h; --sl) eliminate(sl, sl + 1 < a.ns ? sl + 1 : -1, -1);
        if (threadIdx.x == 0) {                                      // this half's pivots, to CTA 0
            unsigned ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(ra) : "r"((unsigned)__cvta_generic_to_shared(&other_bad)));
            asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(ra), "r"(sh.bad) : "memory");
        }
    }
    cluster_sync();
    if (half == 0) {
        eliminate(h, h - 1, h + 1 < a.ns ? h + 1 : -1);
        if (threadIdx.x == 0) *not_spd = sh.bad | other_bad;
    }
    cluster_sync();                                                  // y of the middle slab is the solution there
    auto back = [&](int sl, int next) {
        const int base = sl * b;
        for (int i = threadIdx.x; i < b; i += NTH) z[i] = cs[min(sl, next) * b + i] * y[next * b + i];
        __syncthreads();
        gemv(sl, [&](int i, double v) { y[base + i] += v; });
    };
    if (half == 0) for (int sl = h - 1; sl >= 0; --sl) back(sl, sl + 1);
    else for (int sl = h + 1; sl < a.ns; ++sl) back(sl, sl - 1);
    // ---- outputs: p in box-lexicographic order, outward fluxes on Robin / Dirichlet faces
    for (int c = c_lo + threadIdx.x; c < c_hi; c += NTH) {
        int lc[3];
        box_coords(a, c, lc);
        const int gc = lc[0] + nx * (lc[1] + ny * lc[2]);
        const double yc = y[c];
        p[gc] = yc;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
            for (int hi = 0; hi < 2; ++hi) {
                const bool boundary = hi ? lc[ax] + 1 == a.sz[ax] : lc[ax] == 0;
                if (!boundary) continue;
                const int sd = 2 * ax + hi;
                const int fi = a.side_off[sd] + side_face(a, ax, lc);
                const double ka = K[(long long)ax * N + gc];
                if (a.side_type[sd] == 1) q[fi] = t_robin(area[ax], a.h[ax], ka, beta[fi]) * (yc - g[fi]);
                else if (a.side_type[sd] == 2) q[fi] = 2.0 * ah[ax] * ka * (yc - g[fi]);
                else q[fi] = 0.0;
            }
        }
    }
}

// Device address of the scratch array, looked up once per device (with that
// device current) on the first call there.  In host code the name of a
// __device__ variable is a host-side stand-in, not a device address, so the
// kernel gets the looked-up pointer.  The cached address belongs to the
// device's primary context as it was at that first call: after
// cudaDeviceReset the module is loaded afresh and it is stale, so the entry
// point does not support use after a device reset in the same process.
std::mutex g_mu;
double* g_scratch_ptr[64] = {};

cudaError_t scratch_for_device(int dev, double** ptr) {
    std::lock_guard<std::mutex> lk(g_mu);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!g_scratch_ptr[dev]) {
        double* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress((void**)&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_ptr[dev] = p;
    }
    *ptr = g_scratch_ptr[dev];
    return cudaSuccess;
}

template <int NTH>
cudaError_t launch_box(cudaStream_t st, BoxArgs a, const double* K, const double* f, const double* g,
                       const double* beta, double* p, double* q, double* scratch, int* not_spd) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(NTH);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_box_solve_noalloc<NTH>, a, K, f, g, beta, p, q, scratch, not_spd);
}

}  // namespace

extern "C" mrcm_status mrcm_box_solve_noalloc(const int box[3], const double h[3], const int side_type[6],
                                              const double* K, const double* f, const double* g,
                                              const double* beta, double* p, double* q_out, int* not_spd,
                                              void* stream) {
    if (!box || !h || !side_type || !K || !f || !p || !q_out || !not_spd) return MRCM_ERR_INVALID_ARG;
    BoxArgs a;
    long long nfaces = 0;
    bool any_fixed = false;
    for (int ax = 0; ax < 3; ++ax) {
        if (box[ax] < 1 || !(h[ax] > 0)) return MRCM_ERR_INVALID_ARG;
        a.sz[ax] = box[ax];
        a.h[ax] = h[ax];
    }
    // the fixed scratch bounds the problem: larger boxes are refused, never truncated
    // (the cell count is formed in 64 bits, before any product is narrowed to int)
    if ((long long)box[0] * box[1] * box[2] > kNaMaxCells) return MRCM_ERR_OOM;
    for (int sd = 0; sd < 6; ++sd) {
        if (side_type[sd] < 0 || side_type[sd] > 2) return MRCM_ERR_INVALID_ARG;
        a.side_type[sd] = side_type[sd];
        a.side_off[sd] = (int)nfaces;
        const int ax = sd / 2;
        const int t1 = ax == 0 ? 1 : 0, t2 = ax == 2 ? 1 : 2;
        nfaces += (long long)box[t1] * box[t2];
        if (side_type[sd] != 0) any_fixed = true;
    }
    if (!any_fixed) return MRCM_ERR_INVALID_ARG;          // all sides no-flow: p undetermined
    if (!g || !beta) return MRCM_ERR_INVALID_ARG;
    int sa = 2;
    for (int ax = 1; ax >= 0; --ax) if (box[ax] > box[sa]) sa = ax;
    a.sa = sa;
    a.ua = sa == 0 ? 1 : 0;
    a.va = sa == 2 ? 1 : 2;
    a.su = box[a.ua];
    a.b = box[a.ua] * box[a.va];
    a.ns = box[sa];
    a.N = a.b * a.ns;
    if (a.N > kNaMaxCells || a.b > kNaMaxBlock || (long long)a.ns * a.b * a.b > kNaMaxW) return MRCM_ERR_OOM;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return MRCM_ERR_CUDA;
    double* scratch = nullptr;
    e = scratch_for_device(dev, &scratch);
    if (e != cudaSuccess) return MRCM_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    switch (mrcm::sweep64_threads(a.b)) {
    case 128: e = launch_box<128>(st, a, K, f, g, beta, p, q_out, scratch, not_spd); break;
    case 192: e = launch_box<192>(st, a, K, f, g, beta, p, q_out, scratch, not_spd); break;
    case 352: e = launch_box<352>(st, a, K, f, g, beta, p, q_out, scratch, not_spd); break;
    default: e = launch_box<576>(st, a, K, f, g, beta, p, q_out, scratch, not_spd); break;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? MRCM_OK : MRCM_ERR_CUDA;
}
