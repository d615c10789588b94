// Local solve of the mixed modes with the block products on the tensor cores
// (one launch: the first solve, or the FP64-residual refinement passes), for the
// subdomains whose block factor is stored in fragment order (SubInfo::frag).
// Included by mrcm_local.cu inside its anonymous namespace.
//
// The slab recursion is the one of solve_one (forward Y_s = W_s Z_s, backward
// x_s = Y_s + W_s (t x_{s+1})), built around three things:
//
//   * W streams.  A block is stored as panels of 16 k-columns, each a row of
//     16 x 16 tiles in the order of the MMA's A fragments (frag_off), and one
//     producer warp keeps a ring of panels filled by bulk copies through the whole
//     pass -- over slab and sweep boundaries -- while eight warps consume them
//     (mbarriers full / empty).  Before, a block was fetched whole into one or two
//     buffers between barriers, with one CTA per SM at b >= 128 (or read from L2
//     above 192), and the copy, the FP64 residual and the product took turns.
//   * Products by mma.sync (m16n8k16, BF16): FP32 operands are cut into three BF16
//     pieces (24 bits), the six piece products down to 2^-24 relative are summed
//     per panel in a fresh accumulator and added in FP32 (the tensor core
//     truncates its running sum).  W is cut in registers as it is consumed, Z once
//     per slab by the thread that forms it.
//   * Everything per entry (FP64 residual, Y and X traffic) is done by consecutive
//     threads on consecutive cells; the product's result passes through shared
//     memory (P) once.  Two CTAs per SM overlap one's FP64 with the other's products.
//
// 256 x 256 x 128 cells, uneven blocks of 64 to 256: first solve 11.5 -> 3.8 ms, six
// sweeps 37.8 -> 11.6 ms; 256 x 512 x 128 cells, blocks of 128: 11.0 -> 6.5 and
// 39.5 -> 23.0 ms.  A CTA spends about half of a pass on the entries and a third on the
// products; neither the instructions that cut W (stored ready cut it was no faster) nor
// the chain of the six products bounds it.
#pragma once

constexpr int kBigWarps = 8;                          // consumer warps; one producer warp after them
constexpr int kBigThreads = 32 * (kBigWarps + 1);

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t r[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float d[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (a, b) = p1 + p2 + p3, BF16 pairs (a in the low half)
__device__ __forceinline__ void cut3(float a, float b, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p1) : "f"(b), "f"(a));
    const float a1 = a - __uint_as_float(p1 << 16), b1 = b - __uint_as_float(p1 & 0xFFFF0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p2) : "f"(b1), "f"(a1));
    const float a2 = a1 - __uint_as_float(p2 << 16), b2 = b1 - __uint_as_float(p2 & 0xFFFF0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p3) : "f"(b2), "f"(a2));
}
__device__ __forceinline__ void bar_consumers() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(bar)) : "memory");
}

struct BigArgs {
    LocalArgs g;
    int stages, stage_bytes;
    int ring, zp, p, co, cols, bars;   // shared-memory offsets (BigSmem)
};

// One panel sequence state per thread: the count of panels consumed (produced) so far.
template <bool kSweep, int U>
__global__ void __launch_bounds__(kBigThreads, U <= 2 ? 2 : 1)
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
        const int nt = (b + 15) >> 4, ldp = 16 * nt + 4, zs = 32 * nt + 16;
        const int ncap = (((m + G - 1) / G + 15) >> 4) << 4;   // columns the planes hold
        const uint32_t zpl = (uint32_t)ncap * zs;         // bytes of one piece's plane
        unsigned char* Zp = sm + a.zp;                    // [piece][column][k] BF16
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
        const long long wst = frag_stride(b);
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
            const int npair = (na + 15) >> 4;             // 16-column groups of the products
            if (producer) {
                // ---- W panels W_0 .. W_{ns-1}, W_{ns-2} .. W_0 into the ring
                if (lane == 0) {
                    const uint32_t bytes = (uint32_t)nt * 1024u;
                    for (int q = 0; q < 2 * ns - 1 && !abort_s; ++q) {
                        const float* src = W + (q < ns ? q : 2 * ns - 2 - q) * wst;
                        for (int k = 0; k < nt; ++k) {
                            if (!mbar_wait(&empty[stage], parity ^ 1u)) { abort_s = 1; atomicAdd(&g.status[ST_TIMEOUT], 1); break; }
                            bulk_load(sm + a.ring + stage * a.stage_bytes, src + (long long)k * nt * 256, bytes, &full[stage]);
                            if (++stage == (uint32_t)S) { stage = 0; parity ^= 1u; }
                        }
                    }
                }
                __syncwarp();
                stage = __shfl_sync(0xffffffffu, stage, 0);
                parity = __shfl_sync(0xffffffffu, parity, 0);
            } else {
                // ---- consumers
                for (uint32_t e = tid; e < 3 * zpl / 16; e += 256) reinterpret_cast<uint4*>(Zp)[e] = make_uint4(0u, 0u, 0u, 0u);
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
                // P[column][row] = W_q Z for every 16-row tile and 16-column group: the products of
                // the panels as they arrive, then (after `before_store`) the results
                float acc[U][8];
                auto product = [&]() {
                    const int units = nt * npair;
                    int mi[U], nj[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int x = warp + kBigWarps * u;
                        nj[u] = x < units ? x / nt : -1;
                        mi[u] = x - (x / nt) * nt;
#pragma unroll
                        for (int q = 0; q < 8; ++q) acc[u][q] = 0.0f;
                    }
                    const uint32_t zb = smem_u32(Zp) + (uint32_t)((lane & 7) + ((lane >> 4) & 1) * 8) * zs + ((lane >> 3) & 1) * 16;
                    for (int k = 0; k < nt; ++k) {
                        if (!abort_s && !mbar_wait(&full[stage], parity)) {
                            if (lane == 0) { abort_s = 1; atomicAdd(&g.status[ST_TIMEOUT], 1); }
                        }
                        const unsigned char* pan = sm + a.ring + stage * a.stage_bytes;
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            if (nj[u] < 0) break;
                            const float4* at = reinterpret_cast<const float4*>(pan + mi[u] * 1024) + lane;
                            const float4 w0 = at[0], w1 = at[32];
                            uint32_t af[3][4];
                            cut3(w0.x, w0.y, af[0][0], af[1][0], af[2][0]);
                            cut3(w0.z, w0.w, af[0][1], af[1][1], af[2][1]);
                            cut3(w1.x, w1.y, af[0][2], af[1][2], af[2][2]);
                            cut3(w1.z, w1.w, af[0][3], af[1][3], af[2][3]);
                            uint32_t bf[3][4];
#pragma unroll
                            for (int p = 0; p < 3; ++p) ldsm4(zb + p * zpl + (uint32_t)(16 * nj[u]) * zs + k * 32, bf[p]);
                            float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                            for (int d = 2; d >= 0; --d)
#pragma unroll
                                for (int pa = d; pa >= 0; --pa) {
                                    mma_16816(t0, af[pa], bf[d - pa][0], bf[d - pa][1]);
                                    mma_16816(t1, af[pa], bf[d - pa][2], bf[d - pa][3]);
                                }
#pragma unroll
                            for (int q = 0; q < 4; ++q) { acc[u][q] += t0[q]; acc[u][4 + q] += t1[q]; }
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&empty[stage]);
                        if (++stage == (uint32_t)S) { stage = 0; parity ^= 1u; }
                    }
                };
                auto store_p = [&]() {
                    const int units = nt * npair;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int x = warp + kBigWarps * u;
                        if (x >= units) break;
                        float* q0 = P + (16 * (x / nt) + 2 * (lane & 3)) * ldp + 16 * (x % nt) + (lane >> 2);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            q0[8 * h * ldp] = acc[u][4 * h];
                            q0[(8 * h + 1) * ldp] = acc[u][4 * h + 1];
                            q0[8 * h * ldp + 8] = acc[u][4 * h + 2];
                            q0[(8 * h + 1) * ldp + 8] = acc[u][4 * h + 3];
                        }
                    }
                };
                auto put_z2 = [&](int jj, int i, float za, float zb) {      // cells i (even) and i + 1
                    uint32_t p1, p2, p3;
                    cut3(za, zb, p1, p2, p3);
                    unsigned char* q = Zp + (uint32_t)jj * zs + 2 * i;
                    *reinterpret_cast<uint32_t*>(q) = p1;
                    *reinterpret_cast<uint32_t*>(q + zpl) = p2;
                    *reinterpret_cast<uint32_t*>(q + 2 * zpl) = p3;
                };
                auto particular = [&](int c) {                    // right-hand side of the particular column
                    int lc[3];
                    local_coords(s, c, lc);
                    return g.rhs_dir[s.cell_off + c] + g.f[global_cell(s, lc, g.geo.n)] * vol;
                };
                // entry walk: (column jj, slab cells i, i + 1), consecutive threads on consecutive
                // pairs: the index and address arithmetic, the cut and the stores of Z serve two cells
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
                            float2* pp = reinterpret_cast<float2*>(&P[jj * ldp + i]);
                            if (sl > 0) {
                                const float2 y = *pp;         // Y of the previous slab
                                float* yo = Ys + (g.last_only ? (long long)c : o) - b;
                                yo[0] = y.x;
                                z0 = fmaf(t_s[i], y.x, z0);
                                if (two) { yo[1] = y.y; z1 = fmaf(t_s[i1], y.y, z1); }
                            }
                            const float sb = rsb[jj], n0 = f0 * sb, n1 = f1 * sb;
                            *pp = make_float2(n0 * n0, n1 * n1);    // parked for the column's norm
                            put_z2(jj, i, z0, z1);
                            i += 2 * di;
                            jj += dj;
                            if (i >= 2 * bp) { i -= 2 * bp; ++jj; }
                        }
                    }
                    bar_consumers();
                    if (sl + 1 < ns) stage_load(sl + 1, true);
                    for (int jj = warp; jj < na; jj += kBigWarps) {     // fixed order per column
                        float rr = 0.0f;
                        for (int i = lane; i < b; i += 32) rr += P[jj * ldp + i];
                        for (int o = 16; o > 0; o >>= 1) rr += __shfl_down_sync(0xffffffffu, rr, o);
                        if (lane == 0) nrm[jj] += rr;
                    }
                    product();
                    bar_consumers();                          // the parked norms are read
                    store_p();
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
                        float2 x = *reinterpret_cast<const float2*>(&P[jj * ldp + i]);
                        if (sl + 1 < ns) {
                            const float* y = Ys + (g.last_only ? (long long)(base + i) : o);
                            x.x += y[0];
                            if (two) x.y += y[1];
                        }
                        double* xp = Xs + o;
                        const double x0 = f32_to_f64(x.x * sc_s[i]), x1 = f32_to_f64(x.y * sc_s[i1]);
                        if (kSweep) { xp[0] += x0; if (two) xp[1] += x1; }
                        else { xp[0] = x0; if (two) xp[1] = x1; }
                        if (sl > 0) put_z2(jj, i, t_s[i] * x.x, two ? t_s[i1] * x.y : 0.0f);
                        i += 2 * di;
                        jj += dj;
                        if (i >= 2 * bp) { i -= 2 * bp; ++jj; }
                    }
                    if (sl == 0) break;
                    bar_consumers();
                    stage_load(sl - 1, false);
                    product();
                    store_p();
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
