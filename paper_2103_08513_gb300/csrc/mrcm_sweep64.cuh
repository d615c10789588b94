// In-place inversion of an SPD block in FP64 on register tiles, shared by the
// batched factor kernel and the allocation-free box solve.
//
// The block is held as 4 x 4 tiles of its lower triangle, one tile per thread
// (b <= 128: at most 528 tiles in one CTA; up to 256: at most 2080 tiles over a
// cluster of eight), and swept by the sign-symmetric Gauss-Jordan
// step M[i][j] -= M[i][k] M[k][j] / p (M[i][k] = sigma_i M[k][i], sigma = -1 on
// pivoted indices).
//
// What bounds it: the FP64 units.  A warp's FP64 instruction holds the unit of
// its SM sub-partition for about 64 cycles whatever its active lanes (19 cycles
// per SM over the four), so the count of FP64 warp instructions per pivot is the
// cost: 16 updates and 4 scalings per tile warp -- 60 at b = 50 (64 with the pivot warp's)
// against 40 for the bare triangle; a packed triangle in shared memory with a warp per row took
// about 250 (two operations per entry, idle lanes past the diagonal, a division
// in every warp).  The next pivot and its reciprocal (two FP64 operations, then integer ones)
// are formed by a warp of their own, which at b <= 52 is the fourth
// sub-partition's, while the tile warps update (10 x 10 x 5 box: 440 us with the
// diagonal tile's thread doing it after its updates, 376 us with the warp, 318 us
// once no sign was flipped by an FP64 instruction, 321 us with the integer reciprocal).  2244 blocks of 10 slabs,
// b = 50: 19.3 ms with the packed triangle, 4.3 ms now.
// Blocks above 128 (the tiles no longer fit one SM's registers) are spread over a
// cluster of eight CTAs, tile t on CTA t mod 8; the pivot row goes into every
// CTA's shared memory and the step's barrier is the cluster's (72 x 70 x 48 cells, uneven
// blocks up to 256: 211 ms with a packed triangle in shared or global memory, 25.6 ms).
// 8 x 8 tiles would scale less (72 instead of 80 per 64 entries) but waste more
// on the diagonal and leave one warp per block of 50.
#pragma once
#include <cuda_runtime.h>

#include "mrcm_devmath.cuh"

namespace mrcm {

constexpr int kSw64B = 128;        // largest block of one CTA
constexpr int kSw64BC = 256;       // largest block of a cluster
constexpr int kSw64Cl = 8;         // CTAs of a cluster
constexpr int kSw64T = 4;          // tile edge

// Threads per CTA: whole warps that hold a b x b block (or a cluster's eighth of
// it), one tile each, and the pivot warp (the last one).
__host__ __device__ inline int sweep64_threads(int b) {
    const int nt = (b + kSw64T - 1) / kSw64T, T = nt * (nt + 1) / 2;
    if (b > kSw64B) return T <= 128 * kSw64Cl ? 160 : 320;
    return T <= 96 ? 128 : T <= 160 ? 192 : T <= 320 ? 352 : 576;
}

// Tile (ti >= tj) of thread t.
__device__ __forceinline__ void sweep64_tile(int t, int& ti, int& tj) {
    ti = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (ti * (ti + 1) / 2 > t) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
    tj = t - ti * (ti + 1) / 2;
}

template <int CL>
struct Sweep64Shared {
    double prow[2][CL == 1 ? kSw64B : kSw64BC];        // the pivot row, double-buffered: one barrier per pivot
    double pinv[2];                // 1 / p of the step
    double dnext[2];               // the next pivot's entry before the step's update
    int bad;                       // a pivot was not positive (replaced by 1)
};

// Reciprocal of a pivot; the sign test reads its bits (an FP64 compare would
// add an FP64-unit latency to the pivot chain).
__device__ __forceinline__ double sweep64_pivot(double p, int* bad) {
    const long long u = __double_as_longlong(p);
    if (!(u > 0 && u <= 0x7FF0000000000000ll)) { *bad = 1; p = 1.0; }
    return rcp64(p);
}

template <int CL>
__device__ __forceinline__ void sweep64_barrier() {
    if constexpr (CL == 1) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *dst = v (and dst[1] = w) here, or at the same place in every CTA of the cluster
template <int CL>
__device__ __forceinline__ void sweep64_put(double* dst, double v) {
    if constexpr (CL == 1) { *dst = v; return; }
    const unsigned la = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
    for (int t = 0; t < CL; ++t) {
        unsigned ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(t));
        asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(ra), "d"(v) : "memory");
    }
}
template <int CL>
__device__ __forceinline__ void sweep64_put2(double* dst, double v, double w) {
    if constexpr (CL == 1) { *reinterpret_cast<double2*>(dst) = make_double2(v, w); return; }
    const unsigned la = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
    for (int t = 0; t < CL; ++t) {
        unsigned ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(t));
        asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" :: "r"(ra), "d"(v), "d"(w) : "memory");
    }
}

// a <- inverse of the block whose lower-triangle tiles the threads hold
// (diagonal tiles: both triangles; rows and columns past b are never pivoted).
// Every thread of the CTA (cluster) calls it; `own` marks the threads with a tile
// (not the pivot warp's, the last of each CTA).  The last step's readers of `sh`
// are not waited for.
template <int CL>
__device__ __forceinline__ void sweep64_invert(double (&a)[kSw64T][kSw64T], int ti, int tj, bool own, int b,
                                               Sweep64Shared<CL>& sh) {
    const int i0 = ti * kSw64T, j0 = tj * kSw64T;
    const int nt = (b + kSw64T - 1) / kSw64T;
    const bool pivot_warp = threadIdx.x + 32 >= blockDim.x;
    const bool idle_warp = !__any_sync(0xffffffffu, own);      // no tile: its FP64 instructions would cost all the same
    if (own && ti == 0) sweep64_put<CL>(&sh.pinv[0], sweep64_pivot(a[0][0], &sh.bad));
#pragma unroll 1
    for (int kt = 0; kt < nt; ++kt) {
        const bool rowt = own && ti == kt, colt = own && tj == kt;
#pragma unroll
        for (int kr = 0; kr < kSw64T; ++kr) {
            const int k = kt * kSw64T + kr;
            if (k >= b) break;
            double* pr = sh.prow[kr & 1];
            if (rowt) {                                     // M[k][x], x in or left of the diagonal tile
                sweep64_put2<CL>(pr + j0, a[kr][0], a[kr][1]);
                sweep64_put2<CL>(pr + j0 + 2, a[kr][2], a[kr][3]);
            }
            if (colt && ti > kt) {                          // M[x][k] = M[k][x] below it
                sweep64_put2<CL>(pr + i0, a[0][kr], a[1][kr]);
                sweep64_put2<CL>(pr + i0 + 2, a[2][kr], a[3][kr]);
            }
            if (kr + 1 < kSw64T ? rowt && colt : own && ti == kt + 1 && tj == ti)
                sweep64_put<CL>(&sh.dnext[kr & 1], a[(kr + 1) & 3][(kr + 1) & 3]);
            sweep64_barrier<CL>();
            const double ip = sh.pinv[kr & 1];
            if (pivot_warp) {                               // p_{k+1} as its tile forms it, and its reciprocal
                if (k + 1 < b && (threadIdx.x & 31) == 0) {
                    const double r = pr[k + 1];
                    sh.pinv[(kr + 1) & 1] = sweep64_pivot(fma(-r, r * ip, sh.dnext[kr & 1]), &sh.bad);
                }
                continue;
            }
            if (idle_warp) continue;
            const double2 q0 = reinterpret_cast<const double2*>(pr + j0)[0], q1 = reinterpret_cast<const double2*>(pr + j0)[1];
            const double2 c0 = reinterpret_cast<const double2*>(pr + i0)[0], c1 = reinterpret_cast<const double2*>(pr + i0)[1];
            double rk[4] = {q0.x * ip, q0.y * ip, q1.x * ip, q1.y * ip};
            const double ck[4] = {c0.x, c0.y, c1.x, c1.y};
            if (colt) {                                     // column k rides on the update: -M[i][k] / p
#pragma unroll
                for (int r = 0; r < kSw64T; ++r) a[r][kr] = 0.0;
                rk[kr] = ip;
            }
#pragma unroll
            for (int r = 0; r < kSw64T; ++r) {
                if (r == kr && rowt) {                      // row k: M[k][j] / p, and 1 / p at (k, k)
#pragma unroll
                    for (int c = 0; c < kSw64T; ++c) a[r][c] = rk[c];
                } else {
                    // -M[i][k]; the sign is flipped in its bits (a selected FP64 negation is an FP64 instruction)
                    const double m = __hiloint2double(__double2hiint(ck[r]) ^ (i0 + r < k ? 0 : (int)0x80000000u),
                                                      __double2loint(ck[r]));
#pragma unroll
                    for (int c = 0; c < kSw64T; ++c) a[r][c] = fma(m, rk[c], a[r][c]);
                }
            }
        }
    }
}

// Store the tile and, off the diagonal, its transpose into the full row-major
// b x b matrix W.
__device__ __forceinline__ void sweep64_store(const double (&a)[kSw64T][kSw64T], int ti, int tj, bool own, int b,
                                              double* __restrict__ W) {
    if (!own) return;
    const int i0 = ti * kSw64T, j0 = tj * kSw64T;
#pragma unroll
    for (int r = 0; r < kSw64T; ++r) {
#pragma unroll
        for (int c = 0; c < kSw64T; ++c) {
            const int i = i0 + r, j = j0 + c;
            if (i < b && j < b) {
                W[(long long)i * b + j] = a[r][c];
                if (ti != tj) W[(long long)j * b + i] = a[r][c];
            }
        }
    }
}

}  // namespace mrcm
