// Mixed-precision block factor on the tensor cores for the subdomains with
// fragment-order factors (SubInfo::frag).  Included by mrcm_local.cu inside its
// anonymous namespace.
//
// The block S_s is held as 16 x 16 tiles of its lower triangle (identity past b)
// in the registers of the CTA's warps, in the MMA's accumulator layout, and swept
// 16 pivots at a time with the blocked form of the sign-symmetric Gauss-Jordan
// step.  With P the pivot block, G = M_PP^{-1}, C_i = M_iP, A_i = C_i G and
// sigma_j = -1 on swept blocks:
//   M_ij -= sigma_j A_i C_j^T,   M_iP <- -A_i (i > P),   M_Pj <- -A_j^T (j < P),   M_PP <- G.
// Per step: the pivot row's and column's tiles are published as C_i, the A_i are
// formed (one tile a warp), and every warp updates its tiles, the next diagonal
// tile's warp inverting it (16 FP32 pivots in registers) meanwhile.  Products are m16n8k16 BF16 MMAs on three-piece
// operands (24 bits; six products), summed per step in a fresh accumulator and
// added in FP32: rounding as in the FP32 sweep, pivot block by pivot block.  (The
// variant with the block in tensor memory accumulates there over the whole sweep
// with truncation, which costs the refinement convergence on ill-conditioned blocks.)
//
// What bounds it: per step the chain publish -> A_i -> update and inversion with its
// three barriers, hidden by several CTAs per SM (issue 40 %, shared-memory pipe 51 %,
// tensor pipe 21 % at b = 128).  One FP32 FMA per entry and pivot and a barrier per pivot
// before: 8192 subdomains of 16 slabs, b = 128: 24.6 -> 16.0 ms; 256 x 256 x 128 uneven
// (b 65 .. 256): 17.9 -> 10.0 ms.
#pragma once

constexpr int kFmRow = 48;            // bytes of a 16-column BF16 plane row (padded: conflict-free ldmatrix)
__host__ __device__ inline size_t factor_mma_smem(int b) {
    const size_t nt = (b + 15) / 16;
    return 3 * nt * 16 * kFmRow       // C planes
         + 3 * nt * 512               // A_i as A operands
         + nt * 16 * 17 * 4           // A_i in FP32
         + 2 * 3 * 16 * kFmRow        // G planes (this step's and the next)
         + 3 * 16 * 17 * 4            // M_PP, G (two)
         + 4 * nt * 16 * 4 + 64;      // diagonal, couplings
}

// NW warps of TPW tiles each, the first ND of them diagonal (tile d: warp d mod NW,
// slot d / NW), MINB CTAs per SM.
template <int NW, int TPW, int ND, int MINB>
__global__ void __launch_bounds__(32 * NW, MINB)
k_block_factor_mma(const SubInfo* __restrict__ subs, const int* __restrict__ list, const double* __restrict__ coef,
                   const double* __restrict__ scale, float* __restrict__ Wall, int* __restrict__ status,
                   long long nct, float* __restrict__ scf_all, float* __restrict__ tsc_all) {
    extern __shared__ __align__(128) unsigned char smem_ls[];
    const SubInfo s = subs[list[blockIdx.x]];
    const int b = s.b, su = s.su, nt = (b + 15) >> 4, B = 16 * nt, ntiles = nt * (nt - 1) / 2;
    unsigned char* Cp = smem_ls;                                        // [piece][row][k] BF16
    const uint32_t cpl = (uint32_t)B * kFmRow;
    uint4* Af = reinterpret_cast<uint4*>(Cp + 3 * cpl);                 // [piece][tile][lane]
    float* Ap = reinterpret_cast<float*>(Af + 3 * nt * 32);             // [tile][16][17]
    unsigned char* Gp = reinterpret_cast<unsigned char*>(Ap + nt * 16 * 17);   // [piece][row][k] BF16
    float* D = reinterpret_cast<float*>(Gp + 2 * 3 * 16 * kFmRow);      // [16][17]
    float* Gs = D + 16 * 17;                                            // [2][16][17]
    float* sd = Gs + 2 * 16 * 17;
    float* sup = sd + B;
    float* svp = sup + B;
    float* st = svp + B;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const double* cd = coef + s.cell_off;
    const double* cu = coef + nct + s.cell_off;
    const double* cv = coef + 2 * nct + s.cell_off;
    const double* cs = coef + 3 * nct + s.cell_off;
    const double* sc = scale + s.cell_off;
    float* W = Wall + s.w_off;
    int bad = 0;
    float acc[TPW][8];                       // entry e: row g + 8 ((e >> 1) & 1), column 8 (e >> 2) + 2 t + (e & 1)
    int ti[TPW], tj[TPW];
#pragma unroll
    for (int q = 0; q < TPW; ++q) {
        // the diagonal tiles of this warp, then its share of those below them, row by row
        const int x = q < ND ? 0 : warp + NW * (q - ND), d = warp + NW * q;
        int i = (int)((sqrtf(8.0f * (float)x + 1.0f) - 1.0f) * 0.5f);
        while (i * (i + 1) / 2 > x) --i;
        while ((i + 1) * (i + 2) / 2 <= x) ++i;
        ti[q] = q < ND ? (d < nt ? d : -1) : x < ntiles ? i + 1 : -1;
        tj[q] = q < ND ? d : x - i * (i + 1) / 2;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[q][e] = 0.0f;
    }
    const uint32_t cbase = smem_u32(Cp), gbase = smem_u32(Gp);
    // ldmatrix lane addresses: A operand (rows 0-7 / 8-15, then the upper eight k) and B operand
    // (columns 0-7 with both k halves, then columns 8-15)
    const uint32_t la = (uint32_t)((lane & 7) + ((lane >> 3) & 1) * 8) * kFmRow + ((lane >> 4) & 1) * 16;
    const uint32_t lb = (uint32_t)((lane & 7) + ((lane >> 4) & 1) * 8) * kFmRow + ((lane >> 3) & 1) * 16;
    for (int sl = 0; sl < s.ns; ++sl) {
        const int base = sl * b;
        for (int i = tid; i < B; i += 32 * NW) {
            float d = 1.f, u = 0.f, v = 0.f, tt = 0.f;
            if (i < b) {
                const int c = base + i;
                d = (float)(cd[c] * sc[c] * sc[c]);
                if ((i % su) + 1 < su) u = (float)(-cu[c] * sc[c] * sc[c + 1]);
                if (i + su < b) v = (float)(-cv[c] * sc[c] * sc[c + su]);
                if (sl > 0) tt = (float)(cs[c - b] * sc[c - b] * sc[c]);
                scf_all[s.cell_off + c] = (float)sc[c];
                tsc_all[s.cell_off + c] = sl + 1 < s.ns ? (float)(cs[c] * sc[c] * sc[c + b]) : 0.0f;
            }
            sd[i] = d; sup[i] = u; svp[i] = v; st[i] = tt;
        }
        __syncthreads();
        // S_s = D_s - t o W_{s-1} o t
#pragma unroll
        for (int q = 0; q < TPW; ++q) {
            if (ti[q] < 0) continue;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = 16 * ti[q] + g + 8 * ((e >> 1) & 1), j = 16 * tj[q] + 8 * (e >> 2) + 2 * t + (e & 1);
                float v = -st[i] * st[j] * acc[q][e];        // (t = 0 past b: identity there)
                if (j == i) v += sd[i];
                if (j == i + 1) v += sup[i];
                if (j + 1 == i) v += sup[j];
                if (j == i + su) v += svp[i];
                if (j + su == i) v += svp[j];
                acc[q][e] = v;
            }
        }
        // G = M_PP^{-1} of the diagonal tile that this warp left in D, into buffer `buf`: lane r + 16 h
        // holds columns 8 h .. 8 h + 7 of row r.  The next pivot is formed by every lane from entries
        // fetched before the step's update, so that a pivot's chain is multiply, FMA, reciprocal
        // (an approximation and a Newton step; the IEEE division and a shuffle of the updated pivot
        // took about four times as long).
        auto leave = [&](const float (&v)[8]) {
#pragma unroll
            for (int e = 0; e < 8; ++e) D[(g + 8 * ((e >> 1) & 1)) * 17 + 8 * (e >> 2) + 2 * t + (e & 1)] = v[e];
        };
        auto invert = [&](int buf) {
            __syncwarp();
            const int r = lane & 15, h = lane >> 4;
            float a[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) a[c] = D[r * 17 + 8 * h + c];
            float p = D[0];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int ql = q & 7, qh = q >> 3, nl = (q + 1) & 7, nh = (q + 1) >> 3;
                if (!(p > 0.0f)) { bad = 1; p = 1.0f; }
                float inv;
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(p));
                inv = fmaf(inv, fmaf(-p, inv, 1.0f), inv);
                const float cr = __shfl_sync(0xffffffffu, a[ql], r + 16 * qh);
                if (q < 15) {
                    const float dn = __shfl_sync(0xffffffffu, a[nl], q + 1 + 16 * nh);      // M[q+1][q+1]
                    const float un = __shfl_sync(0xffffffffu, a[nl], q + 16 * nh);          // M[q][q+1]
                    const float ln = __shfl_sync(0xffffffffu, a[ql], q + 1 + 16 * qh);      // M[q+1][q]
                    p = fmaf(-ln, un * inv, dn);
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float rq = __shfl_sync(0xffffffffu, a[c], q + 16 * h) * inv;
                    if (r == q) a[c] = rq; else a[c] = fmaf(-cr, rq, a[c]);
                }
                if (h == qh) a[ql] = r == q ? inv : -cr * inv;
            }
            float* go = Gs + buf * 16 * 17 + r * 17 + 8 * h;
            unsigned char* gq = Gp + buf * 3 * 16 * kFmRow + r * kFmRow + 16 * h;
#pragma unroll
            for (int c = 0; c < 8; c += 2) {
                go[c] = a[c];
                go[c + 1] = a[c + 1];
                uint32_t w[3];
                cut3(a[c], a[c + 1], w[0], w[1], w[2]);
#pragma unroll
                for (int k = 0; k < 3; ++k) *reinterpret_cast<uint32_t*>(gq + k * 16 * kFmRow + 2 * c) = w[k];
            }
        };
        if (warp == 0) { leave(acc[0]); invert(0); }
#pragma unroll 1
        for (int kb = 0; kb < nt; ++kb) {
            const float* Gk = Gs + (kb & 1) * 16 * 17;
            const uint32_t gk = gbase + (kb & 1) * 3 * 16 * kFmRow;
            // (a) publish the C_i
#pragma unroll
            for (int q = ND; q < TPW; ++q) {
                if (ti[q] < 0) continue;
                if (tj[q] == kb) {                     // C_i = M_iP
#pragma unroll
                    for (int h = 0; h < 4; ++h) {             // pairs: (row half h & 1, column half h >> 1)
                        uint32_t p[3];
                        cut3(acc[q][2 * h], acc[q][2 * h + 1], p[0], p[1], p[2]);
                        unsigned char* o = Cp + (16 * ti[q] + g + 8 * (h & 1)) * kFmRow + 16 * (h >> 1) + 4 * t;
#pragma unroll
                        for (int k = 0; k < 3; ++k) *reinterpret_cast<uint32_t*>(o + k * cpl) = p[k];
                    }
                } else if (ti[q] == kb) {                     // C_j = -M_Pj^T
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t p[3];
                        cut3(-acc[q][2 * h], -acc[q][2 * h + 1], p[0], p[1], p[2]);
                        unsigned char* o = Cp + (16 * tj[q] + 8 * (h >> 1) + 2 * t) * kFmRow + 2 * (g + 8 * (h & 1));
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            *reinterpret_cast<unsigned short*>(o + k * cpl) = (unsigned short)p[k];
                            *reinterpret_cast<unsigned short*>(o + k * cpl + kFmRow) = (unsigned short)(p[k] >> 16);
                        }
                    }
                }
            }
            __syncthreads();
            // (b) A_i = C_i G
            for (int i = warp; i < nt; i += NW) {
                if (i == kb) continue;
                uint32_t ca[3][4], gb[3][4];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    ldsm4(cbase + k * cpl + (uint32_t)(16 * i) * kFmRow + la, ca[k]);
                    ldsm4(gk + k * 16 * kFmRow + lb, gb[k]);
                }
                float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int d = 2; d >= 0; --d)
#pragma unroll
                    for (int pa = d; pa >= 0; --pa) {
                        mma_16816(t0, ca[pa], gb[d - pa][0], gb[d - pa][1]);
                        mma_16816(t1, ca[pa], gb[d - pa][2], gb[d - pa][3]);
                    }
                uint32_t w[3][4];                             // the accumulator layout is the A operand's
                cut3(t0[0], t0[1], w[0][0], w[1][0], w[2][0]);
                cut3(t0[2], t0[3], w[0][1], w[1][1], w[2][1]);
                cut3(t1[0], t1[1], w[0][2], w[1][2], w[2][2]);
                cut3(t1[2], t1[3], w[0][3], w[1][3], w[2][3]);
#pragma unroll
                for (int k = 0; k < 3; ++k) Af[(k * nt + i) * 32 + lane] = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
                float* o = Ap + i * 16 * 17 + g * 17 + 2 * t;
                o[0] = t0[0]; o[1] = t0[1]; o[8 * 17] = t0[2]; o[8 * 17 + 1] = t0[3];
                o[8] = t1[0]; o[9] = t1[1]; o[8 * 17 + 8] = t1[2]; o[8 * 17 + 9] = t1[3];
            }
            __syncthreads();
            // (c) the tiles; the next diagonal one first, whose warp then inverts it
#pragma unroll
            for (int q = 0; q < TPW; ++q) {
                if (q == ND && kb + 1 < nt && warp == (kb + 1) % NW) invert((kb + 1) & 1);
                if (ti[q] < 0) continue;
                const int i = ti[q], j = tj[q];
                if (i == kb || j == kb) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int r = g + 8 * ((e >> 1) & 1), c = 8 * (e >> 2) + 2 * t + (e & 1);
                        acc[q][e] = i == j ? Gk[r * 17 + c] : j == kb ? -Ap[i * 16 * 17 + r * 17 + c] : -Ap[j * 16 * 17 + c * 17 + r];
                    }
                    continue;
                }
                uint32_t aw[3][4], cb[3][4];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const uint4 v = Af[(k * nt + i) * 32 + lane];
                    aw[k][0] = v.x; aw[k][1] = v.y; aw[k][2] = v.z; aw[k][3] = v.w;
                    ldsm4(cbase + k * cpl + (uint32_t)(16 * j) * kFmRow + lb, cb[k]);
                }
                float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int d = 2; d >= 0; --d)
#pragma unroll
                    for (int pa = d; pa >= 0; --pa) {
                        mma_16816(t0, aw[pa], cb[d - pa][0], cb[d - pa][1]);
                        mma_16816(t1, aw[pa], cb[d - pa][2], cb[d - pa][3]);
                    }
                const float sg = j < kb ? 1.0f : -1.0f;       // -sigma_j
#pragma unroll
                for (int e = 0; e < 4; ++e) { acc[q][e] = fmaf(sg, t0[e], acc[q][e]); acc[q][4 + e] = fmaf(sg, t1[e], acc[q][4 + e]); }
                if (q < ND && i == kb + 1) leave(acc[q]);
            }
            __syncthreads();                                  // the step's planes are read
        }
        // W_s: every tile and, off the diagonal, its transpose (through this warp's part of the
        // step's shared memory), zero past b
        float* Ws = W + (long long)sl * frag_stride(b);
        float* T = reinterpret_cast<float*>(Cp) + warp * 16 * 17;
#pragma unroll
        for (int q = 0; q < TPW; ++q) {
            if (ti[q] < 0) continue;
            const int i = ti[q], j = tj[q];
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int r = g + 8 * ((e >> 1) & 1), c = 8 * (e >> 2) + 2 * t + (e & 1);
                v[e] = 16 * i + r < b && 16 * j + c < b ? acc[q][e] : 0.0f;
            }
            float4* o = reinterpret_cast<float4*>(Ws + (j * nt + i) * 256) + lane;
            o[0] = make_float4(v[0], v[1], v[2], v[3]);
            o[32] = make_float4(v[4], v[5], v[6], v[7]);
            if (i == j) continue;
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 8; ++e) T[(g + 8 * ((e >> 1) & 1)) * 17 + 8 * (e >> 2) + 2 * t + (e & 1)] = v[e];
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = T[(8 * (e >> 2) + 2 * t + (e & 1)) * 17 + g + 8 * ((e >> 1) & 1)];
            o = reinterpret_cast<float4*>(Ws + (i * nt + j) * 256) + lane;
            o[0] = make_float4(v[0], v[1], v[2], v[3]);
            o[32] = make_float4(v[4], v[5], v[6], v[7]);
        }
        __syncthreads();
    }
    if (__syncthreads_or(bad) && tid == 0) atomicAdd(&status[ST_NOT_SPD], 1);
}
