// In-place inversion of an SPD block in FP64 on register tiles, shared by the
// batched factor kernel and the allocation-free box solve.
//
// The block is held as 4 x 4 tiles of its lower triangle, one tile per thread
// (b <= 128: at most 528 tiles), and swept by the sign-symmetric Gauss-Jordan
// step M[i][j] -= M[i][k] M[k][j] / p (M[i][k] = sigma_i M[k][i], sigma = -1 on
// pivoted indices).
//
// What bounds it: the FP64 units.  A warp's FP64 instruction holds the unit of
// its SM sub-partition for about 64 cycles whatever its active lanes (19 cycles
// per SM over the four), so the count of FP64 warp instructions per pivot is the
// cost: 16 updates and 4 scalings per tile warp -- 60 at b = 50 against 40 for
// the bare triangle; a packed triangle in shared memory with a warp per row took
// about 250 (two operations per entry, idle lanes past the diagonal, a division
// in every warp).  The next pivot and its reciprocal (five dependent operations)
// are formed by a warp of their own, which at b <= 52 is the fourth
// sub-partition's, while the tile warps update (10 x 10 x 5 box: 440 us with the
// diagonal tile's thread doing it after its updates, 376 us with the warp, 318 us
// once no sign was flipped by an FP64 instruction).  2244 blocks of 10 slabs,
// b = 50: 19.3 ms with the packed triangle, 4.5 ms now.
// 8 x 8 tiles would scale less (72 instead of 80 per 64 entries) but waste more
// on the diagonal and leave one warp per block of 50.
#pragma once
#include <cuda_runtime.h>

#include "mrcm_devmath.cuh"

namespace mrcm {

constexpr int kSw64B = 128;        // largest block
constexpr int kSw64T = 4;          // tile edge

// Threads: whole warps that hold a b x b block, one tile each, and the pivot
// warp (the last one); 0 = too large.
__host__ __device__ inline int sweep64_threads(int b) {
    const int nt = (b + kSw64T - 1) / kSw64T, T = nt * (nt + 1) / 2;
    return b > kSw64B ? 0 : T <= 96 ? 128 : T <= 160 ? 192 : T <= 320 ? 352 : 576;
}

// Tile (ti >= tj) of thread t.
__device__ __forceinline__ void sweep64_tile(int t, int& ti, int& tj) {
    ti = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (ti * (ti + 1) / 2 > t) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
    tj = t - ti * (ti + 1) / 2;
}

struct Sweep64Shared {
    double prow[2][kSw64B];        // the pivot row, double-buffered: one barrier per pivot
    double pinv[2];                // 1 / p of the step
    double dnext[2];               // the next pivot's entry before the step's update
    int bad;                       // a pivot was not positive (replaced by 1)
};

// Reciprocal of a pivot; the sign test reads its bits (an FP64 compare would
// add an FP64-unit latency to the pivot chain).
__device__ __forceinline__ double sweep64_pivot(double p, int* bad) {
    const long long u = __double_as_longlong(p);
    if (!(u > 0 && u <= 0x7FF0000000000000ll)) { *bad = 1; p = 1.0; }
    return rcp64c(p);
}

// a <- inverse of the block whose lower-triangle tiles the threads hold
// (diagonal tiles: both triangles; rows and columns past b are never pivoted).
// Every thread of the CTA calls it; `own` marks the threads with a tile (not the
// pivot warp's, the last of the CTA).  The last step's readers of `sh` are not
// waited for.
__device__ __forceinline__ void sweep64_invert(double (&a)[kSw64T][kSw64T], int ti, int tj, bool own, int b,
                                               Sweep64Shared& sh) {
    const int i0 = ti * kSw64T, j0 = tj * kSw64T;
    const int nt = (b + kSw64T - 1) / kSw64T;
    const bool pivot_warp = threadIdx.x + 32 >= blockDim.x;
    if (own && ti == 0) sh.pinv[0] = sweep64_pivot(a[0][0], &sh.bad);
#pragma unroll 1
    for (int kt = 0; kt < nt; ++kt) {
        const bool rowt = own && ti == kt, colt = own && tj == kt;
#pragma unroll
        for (int kr = 0; kr < kSw64T; ++kr) {
            const int k = kt * kSw64T + kr;
            if (k >= b) break;
            double* pr = sh.prow[kr & 1];
            if (rowt) {                                     // M[k][x], x in or left of the diagonal tile
                reinterpret_cast<double2*>(pr + j0)[0] = make_double2(a[kr][0], a[kr][1]);
                reinterpret_cast<double2*>(pr + j0)[1] = make_double2(a[kr][2], a[kr][3]);
            }
            if (colt && ti > kt) {                          // M[x][k] = M[k][x] below it
                reinterpret_cast<double2*>(pr + i0)[0] = make_double2(a[0][kr], a[1][kr]);
                reinterpret_cast<double2*>(pr + i0)[1] = make_double2(a[2][kr], a[3][kr]);
            }
            if (kr + 1 < kSw64T ? rowt && colt : own && ti == kt + 1 && tj == ti)
                sh.dnext[kr & 1] = a[(kr + 1) & 3][(kr + 1) & 3];
            __syncthreads();
            const double ip = sh.pinv[kr & 1];
            if (pivot_warp) {                               // p_{k+1} as its tile forms it, and its reciprocal
                if (k + 1 < b && (threadIdx.x & 31) == 0) {
                    const double r = pr[k + 1];
                    sh.pinv[(kr + 1) & 1] = sweep64_pivot(fma(-r, r * ip, sh.dnext[kr & 1]), &sh.bad);
                }
                continue;
            }
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
