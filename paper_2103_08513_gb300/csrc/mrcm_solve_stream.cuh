// Local solve of the mixed modes for slab blocks above 64 (one launch: the first
// solve, or the FP64-residual refinement passes), for the subdomains with
// SubInfo::stream.  Included by mrcm_local.cu inside its anonymous namespace.
//
// The slab recursion is the one of solve_one (forward Y_s = W_s Z_s, backward
// x_s = Y_s + W_s (t x_{s+1})), built around three things:
//
//   * W streams.  One producer warp keeps a ring of panels (16 rows k of W_s, row
//     major) filled by bulk copies through the whole pass -- over slab and sweep
//     boundaries -- while eight warps consume them (mbarriers full / empty).  Before,
//     a block was fetched whole into one or two buffers between barriers, with one CTA
//     per SM at b >= 128 (or read from L2 above 192), and the copy, the FP64 residual
//     and the product took turns.
//   * Products by FP32 FMAs, a warp's tile of 32 or 16 rows x 4, 8 or 16 columns, k in order:
//     the sums of k_local_solve, bit for bit, so that a column does not depend on the
//     route.  The refinement stops on the residual before a column's last correction,
//     hence the rounding of the correction solve decides what is left in an
//     ill-conditioned column: with factor and products in three BF16 pieces on the
//     tensor cores X of 256 x 512 x 128 cells (sigma 3, stop 1e-10) moved by up to 2.6e-9.
//   * Everything per entry (FP64 residual, Y and X traffic) is done by consecutive
//     threads on consecutive cells; the product's result passes through shared
//     memory (P) once.  Two CTAs per SM overlap one's FP64 with the other's products.
//
// 256 x 256 x 128 cells, uneven blocks of 64 to 256, 13 columns: first solve 11.5 -> 4.3 ms,
// six sweeps 37.8 -> 13.9 ms; 256 x 512 x 128 cells, blocks of 128: 11.0 -> 7.6 and
// 39.5 -> 28.0 ms.  No pipe or memory is near its limit (issue 55 % of the cycles in the first
// solve, 51 % in the sweeps; FMA pipe 26 and 22, FP64 27 in the sweeps, DRAM 31 and 26): the
// entries and the products take turns on the same warps, and at 13 columns half of the warps
// have a tile.  (In three BF16 pieces on the tensor cores 6.5 and 23.0 ms, but see above;
// tiles of 16 rows 9.0 and 32.2, tiles of 8 columns, which give every warp one, 7.7 and 27.8.)
#pragma once

constexpr int kBigWarps = 8;                          // consumer warps; one producer warp after them
constexpr int kBigThreads = 32 * (kBigWarps + 1);

__device__ __forceinline__ void bar_consumers() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(bar)) : "memory");
}

struct BigArgs {
    LocalArgs g;
    int stages, stage_bytes;
    int ring, z, p, co, cols, bars;    // shared-memory offsets (BigSmem)
};

// What a product needs besides the panel sequence.
struct BigProduct {
    const unsigned char* ring;
    unsigned long long *full, *empty;
    int stages, stage_bytes, b, na, ld;
    const float* Z;                    // [column][k]
    float* P;                          // [column][row]
    int* abort_s;
    int* status;
};

// P[column][row] = sum_k W[k][row] Z[column][k] of one slab, the panels as they arrive.  A
// warp takes U tiles of 8 R rows x 4 C columns, lane (rl, cl) of 8 x 4 the rows R rl .. (b a
// multiple of R: one vector load of W; R = 2 with odd b: the rows rl and rl + 8) and the
// columns cl, cl + 4, ...  The lanes that share a row, or a column, are neighbours, which
// makes a load of W one pass of the shared memory and four k of Z two.  With `park` P is
// still read by the others until all consumers are here.
template <int R, int C, int U, bool kOdd>
__device__ __forceinline__ void big_product(const BigProduct& g, bool park, uint32_t& stage, uint32_t& parity) {
    static_assert(R == 4 || R == 2, "rows a lane");
    const int b = g.b, rt = (b + 8 * R - 1) / (8 * R), tiles = rt * ((g.na + 4 * C - 1) / (4 * C));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cl = (lane & 1) | ((lane >> 1) & 2), rl = ((lane >> 1) & 1) | ((lane >> 2) & 6);
    float acc[U][R][C];
    int wo[U], zo[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int x = min(warp + kBigWarps * u, tiles - 1), cb = x / rt, i0 = 8 * R * (x - cb * rt);
        wo[u] = kOdd ? min(i0 + rl, b - 1) : min(i0 + R * rl, b - R);        // (rows past the block: never stored)
        zo[u] = 4 * C * cb + cl;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) acc[u][r][c] = 0.0f;
    }
    const uint32_t zbase = smem_u32(g.Z), rbase = smem_u32(g.ring), b4 = 4u * (uint32_t)b;
    for (int k0 = 0; k0 < b; k0 += 16) {
        if (!mbar_try_wait(&g.full[stage], parity) && !*g.abort_s && !mbar_wait(&g.full[stage], parity)) {
            if (lane == 0) { *g.abort_s = 1; atomicAdd(&g.status[ST_TIMEOUT], 1); }
        }
        const uint32_t pan = rbase + stage * (uint32_t)g.stage_bytes;
        const int rows = min(16, b - k0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (warp + kBigWarps * u >= tiles) break;
            uint32_t zc[C];                                   // shared addresses (32 bits, immediate offsets)
#pragma unroll
            for (int c = 0; c < C; ++c) zc[c] = zbase + 4u * (uint32_t)(min(zo[u] + 4 * c, g.na - 1) * g.ld + k0);
            uint32_t w = pan + 4u * (uint32_t)wo[u];
            const uint32_t w8 = kOdd ? 4u * (uint32_t)(min(wo[u] + 8, b - 1) - wo[u]) : 0u;
            auto load_w = [&](float (&v)[R]) {
                if constexpr (kOdd) {
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(w));
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[1]) : "r"(w + w8));
                } else if constexpr (R == 4) {
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(w));
                } else {
                    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(w));
                }
                w += b4;
            };
            auto group = [&](int k) {
                float z[C][4], v[4][R];
#pragma unroll
                for (int c = 0; c < C; ++c)
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                 : "=f"(z[c][0]), "=f"(z[c][1]), "=f"(z[c][2]), "=f"(z[c][3]) : "r"(zc[c] + 4u * k));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) load_w(v[kk]);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                    for (int c = 0; c < C; ++c)
#pragma unroll
                        for (int r = 0; r < R; ++r) acc[u][r][c] = fmaf(v[kk][r], z[c][kk], acc[u][r][c]);
            };
            if (rows == 16) {
#pragma unroll
                for (int k = 0; k < 16; k += 4) group(k);
            } else {
                int k = 0;
#pragma unroll 1
                for (; k + 4 <= rows; k += 4) group(k);
                if constexpr (R != 4) {                       // (b a multiple of four: none left)
#pragma unroll 1
                    for (; k < rows; ++k) {
                        float v[R];
                        load_w(v);
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            float zz;
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(zz) : "r"(zc[c] + 4u * k));
#pragma unroll
                            for (int r = 0; r < R; ++r) acc[u][r][c] = fmaf(v[r], zz, acc[u][r][c]);
                        }
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&g.empty[stage]);
        if (++stage == (uint32_t)g.stages) { stage = 0; parity ^= 1u; }
    }
    if (park) bar_consumers();
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int x = warp + kBigWarps * u;
        if (x >= tiles) break;
        const int i = 8 * R * (x % rt) + (kOdd ? rl : R * rl);
        if (i >= b) continue;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int jj = zo[u] + 4 * c;
            if (jj >= g.na) break;
            float* q = g.P + jj * g.ld + i;
            if constexpr (kOdd) {
                q[0] = acc[u][0][c];
                if (i + 8 < b) q[8] = acc[u][1][c];
            } else if constexpr (R == 4) {
                *reinterpret_cast<float4*>(q) = make_float4(acc[u][0][c], acc[u][1][c], acc[u][2][c], acc[u][3][c]);
            } else {
                *reinterpret_cast<float2*>(q) = make_float2(acc[u][0][c], acc[u][1][c]);
            }
        }
    }
}

// One panel sequence state per thread: the count of panels consumed (produced) so far.
template <bool kSweep, int U>
__global__ void __launch_bounds__(kBigThreads, U == 1 ? 2 : 1)
k_solve_big(BigArgs a, const float* __restrict__ Wall) {
    extern __shared__ __align__(128) unsigned char smem_ls[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the pass's launch for the smaller blocks may join
    const LocalArgs& g = a.g;
    unsigned char* sm = smem_ls;
    unsigned long long* full = reinterpret_cast<unsigned long long*>(sm + a.bars);
    unsigned long long* empty = full + a.stages;
    __shared__ int item, na_s, abort_s, nbad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool producer = warp == kBigWarps;
    const int S = a.stages;
    if (tid == 0) {
        abort_s = 0;
        for (int q = 0; q < S; ++q) {
            mbar_init(&full[q]);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(&empty[q])), "r"(kBigWarps) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    uint32_t stage = 0, parity = 0;                       // of the next panel
    const int nlist = g.nlist;
    const int G = g.col_groups <= 1 || nlist <= 0 ? 1 : max(1, min(g.col_groups, (int)gridDim.x / nlist));
    const double vol = g.geo.h[0] * g.geo.h[1] * g.geo.h[2];
    for (;;) {
        if (tid == 0) item = atomicAdd(g.queue, 1);
        __syncthreads();
        const int it = item;
        __syncthreads();
        if (it >= nlist * G || abort_s) break;
        const int grp = it % G;
        const SubInfo s = g.subs[g.list[it / G]];
        const int b = s.b, m = s.m, N = s.N, su = s.su, nI = s.nI, ns = s.ns;
        const int nt = (b + 15) >> 4, ld = 16 * nt + 4;
        const int ncap = (((m + G - 1) / G + 7) >> 3) << 3;    // columns that Z and P hold
        float* Z = reinterpret_cast<float*>(sm + a.z);    // [column][k]
        float* P = reinterpret_cast<float*>(sm + a.p);    // [column][row]
        double* co_d = reinterpret_cast<double*>(sm + a.co);
        double* co_u = co_d + b;
        double* co_v = co_u + b;
        double* co_sp = co_v + b;
        double* co_sm = co_sp + b;
        float* t_s = reinterpret_cast<float*>(co_sm + b); // coupling to the previous slab (scaled)
        float* sc_s = t_s + b;
        unsigned* msk_s = reinterpret_cast<unsigned*>(sc_s + b);
        short* fq_s = reinterpret_cast<short*>(msk_s + b);          // [cell][6] face, -1 none
        signed char* fcol_s = reinterpret_cast<signed char*>(fq_s + 6 * b);
        int* cols = reinterpret_cast<int*>(sm + a.cols);
        float* rsb = reinterpret_cast<float*>(cols + ncap);
        float* nrm = rsb + ncap;
        const double* cd = g.coef + s.cell_off;
        const double* cu = g.coef + g.nct + s.cell_off;
        const double* cv = g.coef + 2 * g.nct + s.cell_off;
        const double* cs = g.coef + 3 * g.nct + s.cell_off;
        const float* tsc = g.tsc + s.cell_off;
        const float* scf = g.scf + s.cell_off;
        const float* W = Wall + s.w_off;
        double* Xs = g.X + s.x_off;
        float* Ys = reinterpret_cast<float*>(g.Ybuf) + s.y_off;
        int* conv = g.conv + s.rhs_off;
        const long long wst = wstride<float>(b);
        const int np_pass = kSweep ? max(1, g.passes) : 1;
        for (int ps = 0; ps < np_pass; ++ps) {
            // ---- active columns (deterministic compaction by one warp)
            if (warp == 0) {
                int base = 0;
                for (int j0 = 0; j0 < m; j0 += 32) {
                    const int j = j0 + lane;
                    const bool act = j < m && (!g.last_only || j == m - 1) && (!kSweep || conv[j] == 0) && (G == 1 || j % G == grp);
                    const unsigned bal = __ballot_sync(0xffffffffu, act);
                    if (act) cols[base + __popc(bal & ((1u << lane) - 1u))] = j;
                    base += __popc(bal);
                }
                if (lane == 0) { na_s = base; nbad = 0; }
            }
            __syncthreads();
            const int na = na_s;
            if (na == 0 || abort_s) { __syncthreads(); break; }
            if (producer) {
                // ---- W panels W_0 .. W_{ns-1}, W_{ns-2} .. W_0 into the ring
                if (lane == 0) {
                    const uint32_t whole = 64u * (uint32_t)b, rest = (uint32_t)(4 * wst) - (uint32_t)(nt - 1) * whole;
                    for (int q = 0; q < 2 * ns - 1 && !abort_s; ++q) {
                        const float* src = W + (q < ns ? q : 2 * ns - 2 - q) * wst;
                        for (int k = 0; k < nt; ++k) {
                            if (!mbar_wait(&empty[stage], parity ^ 1u)) { abort_s = 1; atomicAdd(&g.status[ST_TIMEOUT], 1); break; }
                            bulk_load(sm + a.ring + stage * a.stage_bytes, src + 16 * k * b, k + 1 < nt ? whole : rest, &full[stage]);
                            if (++stage == (uint32_t)S) { stage = 0; parity ^= 1u; }
                        }
                    }
                }
                __syncwarp();
                stage = __shfl_sync(0xffffffffu, stage, 0);
                parity = __shfl_sync(0xffffffffu, parity, 0);
            } else {
                // ---- consumers
                for (int e = tid; e < na; e += 256) {
                    nrm[e] = 0.0f;
                    float sc = 1.0f;
                    if (kSweep) {
                        const float bn = (float)g.bnorm[s.rhs_off + cols[e]];
                        if (bn > 0.0f) sc = rsqrtf(bn);
                    }
                    rsb[e] = sc;
                }
                // one slab cell's staged data: loaded ahead (before a product), stored after it
                double pd[5];
                float pt = 0.f, psc = 0.f;
                int pf[3];
                auto stage_load = [&](int sl, bool fwd) {
                    if (tid >= b) return;
                    const int c = sl * b + tid;
                    psc = scf[c];
                    pt = sl > 0 ? tsc[c - b] : 0.0f;
                    if (!fwd) return;
                    const int* fw = reinterpret_cast<const int*>(g.cface + 6 * (s.cell_off + c));
#pragma unroll
                    for (int q = 0; q < 3; ++q) pf[q] = fw[q];
                    if (kSweep) {
                        pd[0] = cd[c]; pd[1] = cu[c]; pd[2] = cv[c];
                        pd[3] = c + b < N ? cs[c] : 0.0;
                        pd[4] = sl > 0 ? cs[c - b] : 0.0;
                    }
                };
                auto stage_store = [&](bool fwd) {
                    if (tid >= b) return;
                    sc_s[tid] = psc;
                    t_s[tid] = pt;
                    if (!fwd) return;
                    if (kSweep) { co_d[tid] = pd[0]; co_u[tid] = pd[1]; co_v[tid] = pd[2]; co_sp[tid] = pd[3]; co_sm[tid] = pd[4]; }
                    const int u = tid % su;
                    unsigned mk = (u + 1 < su ? kNbUp : 0u) | (u > 0 ? kNbUm : 0u) | (tid + su < b ? kNbVp : 0u) | (tid >= su ? kNbVm : 0u);
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const int f = (short)(pf[q >> 1] >> (16 * (q & 1)));
                        const int col = f >= 0 ? g.faces[s.face_off + f].col : -1;
                        fq_s[6 * tid + q] = (short)f;
                        fcol_s[6 * tid + q] = (signed char)col;
                        if (col >= 0) mk |= 1u << (col & 15);
                    }
                    msk_s[tid] = mk;
                };
                const BigProduct bp_ = {sm + a.ring, full, empty, S, a.stage_bytes, b, na, ld, Z, P, &abort_s, g.status};
                auto product = [&](bool park) {
                    // four rows a lane where b allows it and the tiles of 32 rows fit the warps
                    const bool wide = !(b & 3) && (b + 31) / 32 * ((na + 15) / 16) <= kBigWarps * U;
                    if (b & 1) {
                        if (na <= 4) big_product<2, 1, 2, true>(bp_, park, stage, parity);
                        else big_product<2, 4, 2 * U, true>(bp_, park, stage, parity);
                    } else if (!wide) {
                        if (na <= 4) big_product<2, 1, 2, false>(bp_, park, stage, parity);
                        else big_product<2, 4, 2 * U, false>(bp_, park, stage, parity);
                    } else {
                        if (na <= 4) big_product<4, 1, 1, false>(bp_, park, stage, parity);
                        else if (na <= 8) big_product<4, 2, 1, false>(bp_, park, stage, parity);
                        else big_product<4, 4, U, false>(bp_, park, stage, parity);
                    }
                };
                auto particular = [&](int c) {                    // right-hand side of the particular column
                    int lc[3];
                    local_coords(s, c, lc);
                    return g.rhs_dir[s.cell_off + c] + g.f[global_cell(s, lc, g.geo.n)] * vol;
                };
                // entry walk: (column jj, slab cells i, i + 1), consecutive threads on consecutive
                // pairs: the index and address arithmetic and the stores of Z serve two cells
                // (the two entry phases were half of a pass, ~100 instructions a cell)
                const int bp = (b + 1) >> 1;
                const int jj0 = tid / bp, i0 = tid - jj0 * bp, dj = 256 / bp, di = 256 - dj * bp;
                stage_load(0, true);
                stage_store(true);
                bar_consumers();
                // ---- forward sweep
                for (int sl = 0; sl < ns; ++sl) {
                    const int base = sl * b;
                    {
                        int jj = jj0, i = 2 * i0;
                        for (int e = tid; e < na * bp; e += 256) {
                            const int j = cols[jj];
                            const int c = base + i;
                            const bool two = i + 1 < b;
                            const long long o = (long long)j * N + c;
                            const int i1 = two ? i + 1 : i;       // (a lone last cell twice, its second result dropped)
                            const unsigned mk0 = msk_s[i], mk1 = msk_s[i1];
                            double r0 = 0.0, r1 = 0.0;
                            if (j == m - 1) {
                                r0 = particular(c);
                                r1 = two ? particular(c + 1) : 0.0;
                            } else {
                                const int kb = j < nI ? j : j - nI;
                                if (((mk0 | mk1) >> (kb & 15)) & 1u) {
                                    const double* fv = (j < nI ? g.face_tr : g.face_u) + s.face_off;
#pragma unroll
                                    for (int q = 0; q < 6; ++q) {
                                        if (fcol_s[6 * i + q] == kb) r0 = fv[fq_s[6 * i + q]];
                                        if (fcol_s[6 * i1 + q] == kb) r1 = fv[fq_s[6 * i1 + q]];
                                    }
                                }
                            }
                            if (kSweep) {                     // r - A x as one FMA chain each
                                const double* x = Xs + o;
                                const double xa = x[0], xb = two ? x[1] : 0.0;
                                r0 = fma(-co_d[i], xa, r0);
                                if (mk0 & kNbUp) r0 = fma(co_u[i], xb, r0);
                                if (mk0 & kNbUm) r0 = fma(co_u[i - 1], x[-1], r0);
                                if (mk0 & kNbVp) r0 = fma(co_v[i], x[su], r0);
                                if (mk0 & kNbVm) r0 = fma(co_v[i - su], x[-su], r0);
                                if (sl + 1 < ns) r0 = fma(co_sp[i], x[b], r0);
                                if (sl > 0) r0 = fma(co_sm[i], x[-b], r0);
                                if (two) {
                                    r1 = fma(-co_d[i1], xb, r1);
                                    if (mk1 & kNbUp) r1 = fma(co_u[i1], x[2], r1);
                                    if (mk1 & kNbUm) r1 = fma(co_u[i], xa, r1);
                                    if (mk1 & kNbVp) r1 = fma(co_v[i1], x[su + 1], r1);
                                    if (mk1 & kNbVm) r1 = fma(co_v[i1 - su], x[1 - su], r1);
                                    if (sl + 1 < ns) r1 = fma(co_sp[i1], x[b + 1], r1);
                                    if (sl > 0) r1 = fma(co_sm[i1], x[1 - b], r1);
                                }
                            }
                            const float f0 = f64_to_f32_rz(r0), f1 = two ? f64_to_f32_rz(r1) : 0.0f;
                            float z0 = f0 * sc_s[i], z1 = f1 * sc_s[i1];
                            float2* pp = reinterpret_cast<float2*>(&P[jj * ld + i]);
                            if (sl > 0) {
                                const float2 y = *pp;         // Y of the previous slab
                                float* yo = Ys + (g.last_only ? (long long)c : o) - b;
                                yo[0] = y.x;
                                z0 = fmaf(t_s[i], y.x, z0);
                                if (two) { yo[1] = y.y; z1 = fmaf(t_s[i1], y.y, z1); }
                            }
                            const float sb = rsb[jj], n0 = f0 * sb, n1 = f1 * sb;
                            *pp = make_float2(n0 * n0, n1 * n1);    // parked for the column's norm
                            *reinterpret_cast<float2*>(&Z[jj * ld + i]) = make_float2(z0, z1);
                            i += 2 * di;
                            jj += dj;
                            if (i >= 2 * bp) { i -= 2 * bp; ++jj; }
                        }
                    }
                    bar_consumers();
                    if (sl + 1 < ns) stage_load(sl + 1, true);
                    for (int jj = warp; jj < na; jj += kBigWarps) {     // fixed order per column
                        float rr = 0.0f;
                        for (int i = lane; i < b; i += 32) rr += P[jj * ld + i];
                        for (int o = 16; o > 0; o >>= 1) rr += __shfl_down_sync(0xffffffffu, rr, o);
                        if (lane == 0) nrm[jj] += rr;
                    }
                    product(true);                            // (the parked norms are read)
                    if (sl + 1 < ns) stage_store(true);
                    bar_consumers();
                }
                // ---- backward sweep: P holds x of the last slab, then W_s (t x_{s+1})
                for (int sl = ns - 1; sl >= 0; --sl) {
                    const int base = sl * b;
                    int jj = jj0, i = 2 * i0;
                    for (int e = tid; e < na * bp; e += 256) {
                        const bool two = i + 1 < b;
                        const int i1 = two ? i + 1 : i;
                        const long long o = (long long)cols[jj] * N + base + i;
                        float2 x = *reinterpret_cast<const float2*>(&P[jj * ld + i]);
                        if (sl + 1 < ns) {
                            const float* y = Ys + (g.last_only ? (long long)(base + i) : o);
                            x.x += y[0];
                            if (two) x.y += y[1];
                        }
                        double* xp = Xs + o;
                        const double x0 = f32_to_f64(x.x * sc_s[i]), x1 = f32_to_f64(x.y * sc_s[i1]);
                        if (kSweep) { xp[0] += x0; if (two) xp[1] += x1; }
                        else { xp[0] = x0; if (two) xp[1] = x1; }
                        if (sl > 0) *reinterpret_cast<float2*>(&Z[jj * ld + i]) = make_float2(t_s[i] * x.x, two ? t_s[i1] * x.y : 0.0f);
                        i += 2 * di;
                        jj += dj;
                        if (i >= 2 * bp) { i -= 2 * bp; ++jj; }
                    }
                    if (sl == 0) break;
                    bar_consumers();
                    stage_load(sl - 1, false);
                    product(false);
                    stage_store(false);
                    bar_consumers();
                }
                // ---- convergence bookkeeping
                if (kSweep) {
                    if (tid == 0) atomicAdd(reinterpret_cast<unsigned long long*>(g.status + ST_SWEPT), (unsigned long long)na * N);
                    for (int jj = tid; jj < na; jj += 256) {
                        if (nrm[jj] <= (float)g.tol2) conv[cols[jj]] = 1;          // ||r||^2 / ||b||^2 <= tol^2
                        else atomicAdd(&nbad, 1);
                    }
                } else {
                    for (int jj = tid; jj < na; jj += 256) {
                        g.bnorm[s.rhs_off + cols[jj]] = (double)nrm[jj];
                        conv[cols[jj]] = 0;
                    }
                }
            }
            __syncthreads();                                  // X and conv of the pass are visible, shared memory is free
            if (kSweep && tid == 0 && nbad && g.count_unconverged && ps + 1 == np_pass) atomicAdd(&g.status[ST_UNCONVERGED], nbad);
            if (abort_s) break;
        }
    }
    // after a timeout: wait (bounded) for copies still in flight into the ring
    if (abort_s && producer && lane == 0)
        for (int q = 0; q < S; ++q) mbar_wait(&full[q], 0), mbar_wait(&full[q], 1);
}
