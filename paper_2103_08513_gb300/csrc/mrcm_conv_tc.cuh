// Tensor-core kernels of the warm-start network: the fused forward and
// backward-data pass (tcgen05, one launch for all layers) and the weight
// gradients (mma.sync).  Included by mrcm_learned.cu.
//
// FP32 accuracy on BF16 tensor cores.  An FP32 value is cut into three BF16
// pieces x = x1 + x2 + x3 (each the rounded remainder of the ones before);
// weights are BF16 already.  BF16 products are exact in FP32, so
// sum w (x1 + x2 + x3) carries FP32 accuracy with three MMAs, and for the
// weight gradients (both operands FP32) the six products down to 2^-24
// relative do.
//
// Shared-memory layout of activations ("planes"): per piece and chunk of 8
// channels one plane of 16-byte rows, a row per voxel of the zero-padded box.
// Padding is shared: rows of W + 1 voxels, slices of H + 1 rows, one slice
// before and after, so a tap (dz, dy, dx) is the constant row shift
// (dz (H + 1) + dy) (W + 1) + dx and any 8 consecutive voxels are one 128-byte
// core matrix (8 rows x 16 bytes).  That is the tensor core's K-major layout
// without swizzle (rows = voxels: M, 16 bytes = 8 channels: K) at every row
// shift, so an implicit GEMM over the 27 taps reads the planes in place: 128
// consecutive padded voxels are the M rows of a tile, the rows of padding
// voxels are computed and dropped (593 rows for 500 voxels of 5 x 10 x 10).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace mrcm {

constexpr int kTcMaxLayers = 16;
constexpr int kTcThreads = 512;
constexpr int kTcPairs = 5;             // the nine (dz, dy) shifts two by two (first layer)
constexpr size_t kTcSmemMax = 227 * 1024 - 9216;      // dynamic; the kernels' static part stays below 9 KB

// Padded geometry of a D x H x W box.
struct TcGeo {
    int D, H, W, S;
    int wp, hp;             // W + 1, H + 1
    int vp;                 // rows of a plane
    int v0;                 // row of voxel (0, 0, 0); the largest tap shift too
    int tiles;              // 128-row tiles covering the real voxels
    __host__ __device__ TcGeo(int d, int h, int w) : D(d), H(h), W(w), S(d * h * w) {
        wp = w + 1; hp = h + 1;
        vp = (d + 2) * hp * wp + wp + 1;
        v0 = hp * wp + wp + 1;
        tiles = ((d * hp + h) * wp + w - v0 + 1 + 127) / 128;
    }
    __host__ __device__ int shift(int yz) const { return ((yz / 3 - 1) * hp + yz % 3 - 1) * wp; }
    __host__ __device__ int row(int p) const {
        const int z = p / (H * W), r = p - z * H * W, y = r / W;
        return ((z + 1) * hp + y + 1) * wp + (r - y * W) + 1;
    }
    // real voxel of a plane row, or -1
    __device__ int voxel(int r) const {
        const int q = r / wp, x = r - q * wp - 1, z = q / hp - 1, y = q - (z + 1) * hp - 1;
        return (x >= 0 && y >= 0 && z >= 0 && z < D) ? (z * H + y) * W + x : -1;
    }
};

// The three taps of a (dz, dy) row share one MMA: its N = 3 C columns are the C
// output channels for dx = -1, 0, +1, all taken at the shift of dx = 0, so that
// D_dx[v] = sum w(dz, dy, dx) x[v + shift(dz, dy)] and the output of voxel p is
// D_-1[p - 1] + D_0[p] + D_+1[p + 1] (padding rows give 0).  Nine shifts instead
// of 27 taps: an MMA reads its 128 x 16 A tile from shared memory whatever its N,
// and with N = C = 32 that read bounded it (162 x 73 cycles per tile
// and layer with one MMA per tap, 54 x 57 cycles with three).
//
// The first layer has at most 8 input channels: one 8-channel chunk per piece,
// and an MMA (K = 16) takes two shifts, the second one as the second chunk at the
// distance of the two.  Pairs with a positive distance for every box: dy = -1
// with dy = 0; dy = +1 of dz = -1 with dz = 0; the last shift alone (its second
// chunk repeats the first under zero weights).  Shifts are numbered
// 3 (dz + 1) + dy + 1.
__host__ __device__ inline void tc_pair(int q, int* t0, int* t1) {
    if (q < 3) { *t0 = 3 * q; *t1 = 3 * q + 1; }
    else if (q == 3) { *t0 = 2; *t1 = 5; }
    else { *t0 = 8; *t1 = -1; }
}

// Layer kinds: first (<= 8 channels -> C), hidden (C -> C), output (C -> 1).
enum { kTcFirst = 0, kTcHidden = 1, kTcOut = 2 };
__host__ __device__ inline uint32_t tc_weight_bytes(int kind, int C) {
    return kind == kTcFirst ? (uint32_t)kTcPairs * 3 * C * 32 : kind == kTcHidden ? 27u * (C / 16) * C * 32 : (uint32_t)(C / 16) * 1024;
}
// dynamic shared memory: planes, 128 + largest shift rows of slack (the last tile
// reads past the last plane), weights or the output layer's per-tap sums
__host__ __device__ inline uint32_t tc_plane_bytes(const TcGeo& g, int C) {
    const uint32_t rows = 3u * (C / 8) * g.vp + (uint32_t)max(0, g.v0 + 128 * g.tiles + g.v0 - g.vp);
    return (rows * 16 + 127) & ~127u;
}
__host__ __device__ inline uint32_t tc_wregion_bytes(const TcGeo& g, int C) {
    const uint32_t w = tc_weight_bytes(kTcHidden, C), p = 27u * g.S * 4;
    return ((w > p ? w : p) + 127) & ~127u;
}

struct TcLayer {
    int kind, cin, cout;    // real channels
    uint32_t w_off;         // byte offset of the packed weights
    const float* bias;      // forward: added before the activation; NULL: none
    const float* mask;      // backward: leaky-ReLU derivative of this activation, [b][cout][S]; NULL: none
    float* out;             // FP32 result [b][cout][S] in global memory, or NULL
    int leaky;              // apply the leaky ReLU
    int last;               // nothing follows: no planes written
};
struct TcNet {
    int D, H, W, layers, batch;
    const float* x;         // [b][cin][S]
    const unsigned char* wpack;
    TcLayer l[kTcMaxLayers];
};

// Weights of all layers in the layout of the B operand (K-major core matrices of
// 8 columns x 8 input channels, 128 bytes each; per shift and 16 channels of K:
// [K chunk][N group], N = dx and output channel).  flip: the backward-data layers (input and output
// channels exchanged, taps mirrored; l[i] then holds the exchanged counts).
struct TcPack { int layers, C, flip; int kind[kTcMaxLayers], cin[kTcMaxLayers], cout[kTcMaxLayers]; long long w[kTcMaxLayers]; uint32_t off[kTcMaxLayers]; };
__global__ void __launch_bounds__(256) k_tc_pack(TcPack a, const __nv_bfloat16* __restrict__ w, unsigned char* __restrict__ dst) {
    const int l = blockIdx.y;
    const int kind = a.kind[l], ci = a.cin[l], co = a.cout[l], C = a.C;
    const int N = kind == kTcOut ? 32 : 3 * C;
    const int total = (int)(tc_weight_bytes(kind, C) / 2);
    __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(dst + a.off[l]);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int blk = e / (N * 16), r = e - blk * (N * 16);          // one K = 16 block
        const int kc = r / (N * 8), n = (r / 8) % N, k8 = r & 7;
        int tap = -1, k = 0, m = n;
        if (kind == kTcFirst) { int t0, t1; tc_pair(blk, &t0, &t1); tap = kc ? t1 : t0; k = k8; }
        else if (kind == kTcHidden) { tap = blk / (C / 16); k = (blk % (C / 16)) * 16 + kc * 8 + k8; }
        if (kind != kTcOut) { tap = tap < 0 ? -1 : 3 * tap + n / C; m = n % C; }   // column group = dx
        if (kind == kTcOut) { k = blk * 16 + kc * 8 + k8; tap = n < 27 ? n : -1; m = 0; }
        __nv_bfloat16 v = __float2bfloat16_rn(0.0f);
        if (tap >= 0 && k < ci && m < co)
            v = a.flip ? w[a.w[l] + ((long long)k * co + m) * 27 + 26 - tap] : w[a.w[l] + ((long long)m * ci + k) * 27 + tap];
        d[e] = v;
    }
}

__device__ __forceinline__ uint32_t tcs_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool tcs_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// bounded wait (about two seconds)
__device__ __forceinline__ bool tcs_wait(uint32_t bar, uint32_t parity) {
    if (tcs_try(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (tcs_try(bar, parity)) return true;
        if (clock64() - t0 > 4000000000LL) return false;
    }
}
__device__ __forceinline__ void tcs_sync() {      // block barrier that also orders tcgen05 operations
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// matrix descriptor without its start address: K-chunk stride, 8-row-group stride (bytes)
__device__ __forceinline__ uint64_t tcs_desc(uint32_t lbo, uint32_t sbo) {
    return ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ void tcs_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 :: "r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// 16 accumulator columns of this lane's row; the values are valid after tcs_ld_wait
__device__ __forceinline__ void tcs_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
}
// (the registers pass through the wait, so that no use moves before it)
__device__ __forceinline__ void tcs_ld_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :: "memory");
}
// three BF16 pieces of two values, packed (first value in the low half)
__device__ __forceinline__ void tcs_split(float a, float b, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
    const __nv_bfloat162 h1 = __floats2bfloat162_rn(a, b);
    const float2 f1 = __bfloat1622float2(h1);
    const float a1 = a - f1.x, b1 = b - f1.y;
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(a1, b1);
    const float2 f2 = __bfloat1622float2(h2);
    const __nv_bfloat162 h3 = __floats2bfloat162_rn(a1 - f2.x, b1 - f2.y);
    p1 = *reinterpret_cast<const uint32_t*>(&h1);
    p2 = *reinterpret_cast<const uint32_t*>(&h2);
    p3 = *reinterpret_cast<const uint32_t*>(&h3);
}
// eight channel values of one voxel into the three pieces' planes (row r of chunk c)
__device__ __forceinline__ void tcs_put8(unsigned char* planes, uint32_t pitch, int kc, int c, int r, const float* v) {
    uint4 q1, q2, q3;
    tcs_split(v[0], v[1], q1.x, q2.x, q3.x);
    tcs_split(v[2], v[3], q1.y, q2.y, q3.y);
    tcs_split(v[4], v[5], q1.z, q2.z, q3.z);
    tcs_split(v[6], v[7], q1.w, q2.w, q3.w);
    *reinterpret_cast<uint4*>(planes + (size_t)c * pitch + (size_t)r * 16) = q1;
    *reinterpret_cast<uint4*>(planes + (size_t)(kc + c) * pitch + (size_t)r * 16) = q2;
    *reinterpret_cast<uint4*>(planes + (size_t)(2 * kc + c) * pitch + (size_t)r * 16) = q3;
}

// All MMAs of one 128-row tile (piece 3, the smallest, first), straight-line: the
// A descriptors' low words (row offset, chunk stride) come from a table, the B
// ones step by constants, so that an MMA costs its thread a handful of
// instructions (computing shifts in a loop cost about as long as the MMA itself).
template <int N, int C, int kKind>
__device__ __forceinline__ void tcs_issue(uint32_t d, uint32_t r0, uint64_t bd, const uint2* aoff) {
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (8u << 24);
    constexpr int per = kKind == kTcHidden ? 9 * (C / 16) : kKind == kTcFirst ? kTcPairs : C / 16;    // per piece
    const uint2* tab = aoff + (kKind == kTcHidden ? 0 : kKind == kTcFirst ? 27 * (C / 16) : 27 * (C / 16) + 3 * kTcPairs);
#pragma unroll 1
    for (int pc = 0; pc < 3; ++pc) {
#pragma unroll
        for (int q = 0; q < per; ++q) {
            const uint2 o = tab[pc * per + q];
            tcs_mma(d, ((uint64_t)(o.y | (1u << 14)) << 32) | (o.x + r0), bd + (uint32_t)(q * N * 2), idesc, (uint32_t)(pc | q));
        }
    }
}

// All layers of the network (or of its backward-data pass) on one sample per CTA
// at a time, persistent over the batch: the activations never leave shared
// memory, except the copies a training step needs (TcLayer::out).  Per layer one
// thread issues the MMAs of all tiles (piece 3, the smallest, first), then every
// thread takes one accumulator row through bias, activation and split back into
// the planes.  The output layer computes per-tap sums P[voxel][tap] (taps as the
// 27 columns, 6 MMAs a tile instead of 162) and adds the 27 shifted entries.
//
// What bounds it: the MMAs (54 x 5 per hidden layer and 5 x 10 x 10 sample), which
// the epilogue does not overlap (it rewrites the planes they read): 57 cycles each,
// the 7 KB of operands they read from shared memory.  256 samples (two rounds on
// 152 SMs), four layers of 32 channels: 78 us, against 405 us for four launches of
// SIMT and mma.sync kernels that cut every value 27 times.
template <int C>
__global__ void __launch_bounds__(kTcThreads, 1) k_tc_net(const __grid_constant__ TcNet net) {
    extern __shared__ __align__(128) unsigned char tcsm[];
    constexpr int KC = C / 8;
    const TcGeo g(net.D, net.H, net.W);
    const uint32_t pitch = (uint32_t)g.vp * 16;
    unsigned char* planes = tcsm;
    unsigned char* wreg = tcsm + tc_plane_bytes(g, C);
    __shared__ uint32_t tmem_s;
    __shared__ __align__(8) unsigned long long bars[2];        // MMAs done, weights staged
    // per 32-row segment (a warp's accumulator lanes): D_-1 of the row before its
    // first, D_+1 of the row after its last
    constexpr int kSeg = 4 * (512 / (3 * C));
    __shared__ __align__(16) float edge_lo[kSeg + 1][C], edge_hi[kSeg + 1][C], s_bias[C];
    __shared__ short s_vox[32 * kSeg];                          // the real voxel of each tile row, or -1
    for (int e = threadIdx.x; e < 128 * g.tiles; e += kTcThreads) s_vox[e] = (short)g.voxel(g.v0 + e);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t bmma = tcs_u32(&bars[0]), bw = tcs_u32(&bars[1]);
    uint32_t ncols = 32;
    while (ncols < 3u * C * g.tiles) ncols <<= 1;               // accumulator columns (a power of two)
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(tcs_u32(&tmem_s)), "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bmma), "r"(min(g.tiles, kTcThreads / 32)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bw) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // row offsets (low descriptor words) of the MMAs' A tiles, and the chunk distances of the first layer
    __shared__ uint2 s_aoff[3 * 9 * (C / 16) + 3 * kTcPairs + 3 * (C / 16)];
    for (int e = tid; e < 3 * 9 * (C / 16); e += kTcThreads) {
        const int pc = 2 - e / (9 * (C / 16)), r = e % (9 * (C / 16)), yz = r / (C / 16), k16 = r % (C / 16);
        s_aoff[e] = make_uint2((uint32_t)((pc * KC + 2 * k16) * g.vp + g.shift(yz)) + (((uint32_t)g.vp) << 16), 128u >> 4);
    }
    for (int e = tid; e < 3 * kTcPairs; e += kTcThreads) {
        const int pc = 2 - e / kTcPairs, q = e % kTcPairs;
        int t0, t1;
        tc_pair(q, &t0, &t1);
        const int s0 = g.shift(t0), dist = t1 < 0 ? 0 : g.shift(t1) - s0;
        s_aoff[27 * (C / 16) + e] = make_uint2((uint32_t)(pc * KC * g.vp + s0) + ((uint32_t)dist << 16), 128u >> 4);
    }
    for (int e = tid; e < 3 * (C / 16); e += kTcThreads) {
        const int pc = 2 - e / (C / 16), k16 = e % (C / 16);
        s_aoff[27 * (C / 16) + 3 * kTcPairs + e] = make_uint2((uint32_t)((pc * KC + 2 * k16) * g.vp) + (((uint32_t)g.vp) << 16), 128u >> 4);
    }
    for (uint32_t e = tid; e < tc_plane_bytes(g, C) / 16; e += kTcThreads)      // padding rows stay zero
        reinterpret_cast<uint4*>(planes)[e] = make_uint4(0u, 0u, 0u, 0u);
    tcs_sync();
    const uint32_t tmem = tmem_s;
    uint32_t ph_m = 0, ph_w = 0;
    bool dead = false;                                          // a wait gave up: the rest is marked NaN
    bool w_pending = false;                                     // thread 0: a weight copy not yet waited for
    auto load_w = [&](int l) {                                  // thread 0, weight region free
        const uint32_t bytes = tc_weight_bytes(net.l[l].kind, C);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bw), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     :: "r"(tcs_u32(wreg)), "l"(net.wpack + net.l[l].w_off), "r"(bytes), "r"(bw) : "memory");
        w_pending = true;
    };
    for (int b = blockIdx.x; b < net.batch && !dead; b += gridDim.x) {
        if (tid == 0) load_w(0);
        {   // the sample's input channels into chunk 0
            const int ci = net.l[0].cin;
            const float* xb = net.x + (long long)b * ci * g.S;
            for (int p = tid; p < g.S; p += kTcThreads) {
                float v[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = c < ci ? xb[(long long)c * g.S + p] : 0.0f;
                tcs_put8(planes, pitch, KC, 0, g.row(p), v);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tcs_sync();
        for (int l = 0; l < net.layers; ++l) {
            const TcLayer& L = net.l[l];
            const int kind = L.kind;
            if (lane == 0) {                                    // warp w issues the MMAs of the tiles w, w + 16, ...
                bool ready = warp >= g.tiles || tcs_wait(bw, ph_w);    // (else: no commit, the wait below gives up)
                if (tid == 0) w_pending = !ready;
                const uint64_t bd = (kind == kTcOut ? tcs_desc(32 * 16, 128) : tcs_desc(3 * C * 16, 128)) | (tcs_u32(wreg) >> 4);
                for (int t = warp; ready && t < g.tiles; t += kTcThreads / 32) {
                    const uint32_t r0 = (tcs_u32(planes) >> 4) + (uint32_t)(g.v0 + 128 * t);
                    if (kind == kTcHidden) tcs_issue<3 * C, C, kTcHidden>(tmem + 3u * C * t, r0, bd, s_aoff);
                    else if (kind == kTcFirst) tcs_issue<3 * C, C, kTcFirst>(tmem + 3u * C * t, r0, bd, s_aoff);
                    else tcs_issue<32, C, kTcOut>(tmem + 32u * t, r0, bd, s_aoff);
                }
                if (ready && warp < g.tiles)
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bmma) : "memory");
            }
            __syncwarp();                                       // the issuing thread's warp does not spin beside it
            const bool tout = !tcs_wait(bmma, ph_m);
            ph_w ^= 1u;
            ph_m ^= 1u;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (__syncthreads_or(tout)) { dead = true; break; }
            if (tid == 0 && l + 1 < net.layers) load_w(l + 1);            // the MMAs have read the weights
            const int quarter = warp & 3;
            if (kind == kTcOut) {
                // P[voxel][tap], then the sum over the taps and the logistic
                float* P = reinterpret_cast<float*>(wreg);
                for (int t = warp >> 2; t < g.tiles; t += kTcThreads / 128) {
                    uint32_t lo[16], hi[16];
                    __syncwarp();
                    const uint32_t ta = tmem + 32u * t + ((uint32_t)(32 * quarter) << 16);
                    tcs_ld16(ta, lo);
                    tcs_ld16(ta + 16, hi);
                    tcs_ld_wait(lo);
                    tcs_ld_wait(hi);
                    const int p = s_vox[128 * t + 32 * quarter + lane];
                    if (p >= 0) {
#pragma unroll
                        for (int q = 0; q < 27; ++q) P[p * 27 + q] = __uint_as_float(q < 16 ? lo[q] : hi[q - 16]);
                    }
                }
                tcs_sync();
                const float bias = L.bias[0];
                for (int p = tid; p < g.S; p += kTcThreads) {
                    const int z = p / (g.H * g.W), r = p - z * g.H * g.W, y = r / g.W, x = r - y * g.W;
                    float s = 0.0f;
#pragma unroll
                    for (int q = 0; q < 27; ++q) {
                        const int dz = q / 9 - 1, dy = (q / 3) % 3 - 1, dx = q % 3 - 1;
                        if (z + dz >= 0 && z + dz < g.D && y + dy >= 0 && y + dy < g.H && x + dx >= 0 && x + dx < g.W)
                            s += P[(p + (dz * g.H + dy) * g.W + dx) * 27 + q];
                    }
                    L.out[(long long)b * g.S + p] = 1.0f / (1.0f + __expf(-(s + bias)));
                }
                tcs_sync();                                     // P is overwritten by the next sample's weights
                continue;
            }
            // tasks (tile, 16 channels) over the four warps of an accumulator-lane quarter
            for (int k = warp >> 2; k < g.tiles * (C / 16); k += kTcThreads / 128) {   // the segments' edge rows
                const int t = k / (C / 16), h = k % (C / 16), seg = 4 * t + quarter;
                const uint32_t ta = tmem + (uint32_t)(3 * C * t) + ((uint32_t)(32 * quarter) << 16);
                {
                    uint32_t lo[16], hi[16];
                    __syncwarp();                               // the loads are warp-collective
                    tcs_ld16(ta + 16u * h, lo);
                    tcs_ld16(ta + 2u * C + 16u * h, hi);
                    tcs_ld_wait(lo);
                    tcs_ld_wait(hi);
                    if (lane == 31) {
#pragma unroll
                        for (int c = 0; c < 16; c += 4)
                            *reinterpret_cast<uint4*>(&edge_lo[seg + 1][16 * h + c]) = make_uint4(lo[c], lo[c + 1], lo[c + 2], lo[c + 3]);
                    }
                    if (lane == 0) {
#pragma unroll
                        for (int c = 0; c < 16; c += 4)
                            *reinterpret_cast<uint4*>(&edge_hi[seg][16 * h + c]) = make_uint4(hi[c], hi[c + 1], hi[c + 2], hi[c + 3]);
                    }
                }
            }
            if (tid < C) {
                edge_lo[0][tid] = edge_hi[4 * g.tiles][tid] = 0.0f;
                s_bias[tid] = L.bias && tid < L.cout ? L.bias[tid] : 0.0f;
            }
            __syncthreads();
            const float leak = L.leaky ? 0.01f : 1.0f;         
            for (int k = warp >> 2; k < g.tiles * (C / 16); k += kTcThreads / 128) {
                const int t = k / (C / 16), h = k % (C / 16), seg = 4 * t + quarter, row = g.v0 + 32 * seg + lane;
                const uint32_t ta = tmem + (uint32_t)(3 * C * t) + ((uint32_t)(32 * quarter) << 16);
                const int p = s_vox[32 * seg + lane];
                // the edge lanes take their neighbour from shared memory, the others by a shuffle
                const float* el = edge_lo[lane == 31 ? seg + 1 : seg];
                const float* eh = edge_hi[lane == 0 ? seg : seg + 1];
                {
                    uint32_t lo[16], md[16], hi[16];
                    float v[16];
                    __syncwarp();
                    tcs_ld16(ta + 16u * h, lo);
                    tcs_ld16(ta + (uint32_t)C + 16u * h, md);
                    tcs_ld16(ta + 2u * C + 16u * h, hi);
                    tcs_ld_wait(lo);
                    tcs_ld_wait(md);
                    tcs_ld_wait(hi);
#pragma unroll
                    for (int c4 = 0; c4 < 16; c4 += 4) {
                        const float4 a4 = *reinterpret_cast<const float4*>(el + 16 * h + c4);
                        const float4 z4 = *reinterpret_cast<const float4*>(eh + 16 * h + c4);
                        const float4 b4 = *reinterpret_cast<const float4*>(s_bias + 16 * h + c4);
                        const float aa[4] = {a4.x, a4.y, a4.z, a4.w}, zz[4] = {z4.x, z4.y, z4.z, z4.w}, bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int c = c4 + q;
                            const float up = __shfl_up_sync(0xffffffffu, __uint_as_float(lo[c]), 1);
                            const float dn = __shfl_down_sync(0xffffffffu, __uint_as_float(hi[c]), 1);
                            const float x = ((lane == 0 ? aa[q] : up) + (lane == 31 ? zz[q] : dn)) + __uint_as_float(md[c]) + bb[q];
                            v[c] = x > 0.0f ? x : leak * x;
                        }
                    }
                    if (p >= 0) {
                        const long long o = ((long long)b * L.cout + 16 * h) * g.S + p;
                        if (L.mask) {                           // backward: the derivative of the layer's leaky ReLU
                            float m[16];
#pragma unroll
                            for (int c = 0; c < 16; ++c) m[c] = 16 * h + c < L.cout ? L.mask[o + (long long)c * g.S] : 1.0f;
#pragma unroll
                            for (int c = 0; c < 16; ++c) if (!(m[c] > 0.0f)) v[c] *= 0.01f;
                        }
                        if (L.out) {
#pragma unroll
                            for (int c = 0; c < 16; ++c) if (16 * h + c < L.cout) L.out[o + (long long)c * g.S] = v[c];
                        }
                        if (!L.last) {
                            tcs_put8(planes, pitch, KC, 2 * h, row, v);
                            tcs_put8(planes, pitch, KC, 2 * h + 1, row, v + 8);
                        }
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tcs_sync();
        }
        if (dead)                                               // never a plausible result after a timeout
            for (int bb = b; bb < net.batch; bb += gridDim.x) {
                const TcLayer& L = net.l[net.layers - 1];
                if (L.out)
                    for (int e = tid; e < L.cout * g.S; e += kTcThreads)
                        L.out[(long long)bb * L.cout * g.S + e] = __int_as_float(0x7FC00000);
            }
    }
    if (tid == 0 && w_pending) tcs_wait(bw, ph_w);              // a copy still in flight after a timeout
    tcs_sync();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(ncols));
}

// ---------------------------------------------------------------------------
// Weight gradients: gw[co][ci][tap] = sum_{b, p} g[b][co][p] in[b][ci][p + tap],
// a GEMM of 27 shifted products over K = batch x voxels.  Work items are slabs of
// a sample (zc slices); the item's g and in (with its halo) are cut into planes
// and each of 27 warps (one per tap) accumulates its MT x 16 by NT x 8 channels in
// registers over all items of its CTA (mma.sync m16n8k16 on transposed ldmatrix
// loads: K = voxels are the planes' rows, so a tap is a row shift here too).  The
// CTAs' partial sums are added in a fixed order by k_tc_sum.
//
// What bounds it: the MMAs, six per product of FP32 operands, at the 4 cycles per
// SM that mma.sync takes for m16n8k16 here: 256 samples of 5 x 10 x 10, 32 -> 32
// channels 157 us (136 us of MMAs), against 2480 us for a CTA per channel pair that
// read both arrays 27 times through L1.
// ---------------------------------------------------------------------------
constexpr int kWgThreads = 27 * 32;
__host__ __device__ inline uint32_t wg_smem(int H, int W, int zc, int mt, int nt) {
    const uint32_t xr = (uint32_t)((zc + 2) * (H + 1) * (W + 1) + W + 2), gr = (uint32_t)((zc * H * W + 15) & ~15);
    return 16u * 3u * (xr * nt + gr * 2 * mt) + 4u * gr;
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t r[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t addr, uint32_t r[2]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void wg_mma(float d[4], const uint32_t a[4], const uint32_t b0, const uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One K step: acc[j] += A x (columns of chunk j), the six piece products smallest
// first into a fresh accumulator, which is then added in FP32: the tensor core
// truncates its running sum, and over the hundreds of steps of a batch that bias
// reached 6e-6 of the result; here it is one step's.
template <int NT>
__device__ __forceinline__ void wg_step(float (&acc)[NT][4], const uint32_t (&af)[3][4], uint32_t xbase, uint32_t xrows,
                                        uint32_t xr, int lane) {
    constexpr int J = NT == 1 ? 1 : 2;
#pragma unroll
    for (int j = 0; j < NT; j += J) {
        uint32_t bf[3][2 * J];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            if constexpr (J == 1) ldsm2t(xbase + 16u * ((uint32_t)p * xrows + xr), bf[p]);
            else ldsm4t(xbase + 16u * ((uint32_t)(p * NT + j + (lane >> 4)) * xrows + xr), bf[p]);
        }
#pragma unroll
        for (int jj = 0; jj < J; ++jj) {
            float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int d = 2; d >= 0; --d)
#pragma unroll
                for (int pa = d; pa >= 0; --pa) wg_mma(t, af[pa], bf[d - pa][2 * jj], bf[d - pa][2 * jj + 1]);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[j + jj][q] += t[q];
        }
    }
}

template <int MT, int NT>
__global__ void __launch_bounds__(kWgThreads, 1)
k_tc_wgrad(int D, int H, int W, int zc, int batch, int Cin, int Cout, const float* __restrict__ gsrc,
           const float* __restrict__ in, float* __restrict__ part) {
    extern __shared__ __align__(128) unsigned char tcsm[];
    const int wp = W + 1, hp = H + 1, S = D * H * W, HW = H * W;
    const int xrows = (zc + 2) * hp * wp + wp + 1, grows = (zc * HW + 15) & ~15;
    unsigned char* xp = tcsm;                                   // [piece][NT chunks][xrows] x 16 bytes
    unsigned char* gp = xp + 16u * 3u * NT * xrows;             // [piece][2 MT chunks][grows] x 16 bytes
    int* xrow = reinterpret_cast<int*>(gp + 16u * 3u * 2 * MT * grows);   // x-plane row of each g row
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nz = (D + zc - 1) / zc, items = batch * nz;
    float acc[MT][NT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    for (int e = tid; e < 3 * NT * xrows; e += kWgThreads) reinterpret_cast<uint4*>(xp)[e] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = tid; e < grows; e += kWgThreads) {             // rows past the slab repeat the first voxel (g is zero there)
        const int q = e < zc * HW ? e : 0, z = q / HW, r = q - z * HW, y = r / W;
        xrow[e] = ((z + 1) * hp + y + 1) * wp + (r - y * W) + 1;
    }
    const int shift = ((warp / 9 - 1) * hp + (warp / 3) % 3 - 1) * wp + warp % 3 - 1;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int b = it / nz, z0 = (it - b * nz) * zc, z1 = min(D, z0 + zc), ng = (z1 - z0) * HW;
        __syncthreads();                                        // the previous item's planes are read
        for (int e = tid; e < 2 * MT * grows; e += kWgThreads) {
            const int c = e / grows, q = e - c * grows;
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int co = 8 * c + k;
                v[k] = q < ng && co < Cout ? gsrc[((long long)b * Cout + co) * S + z0 * HW + q] : 0.0f;
            }
            tcs_put8(gp, 16u * grows, 2 * MT, c, q, v);
        }
        const int nx = (zc + 2) * HW;
        for (int e = tid; e < NT * nx; e += kWgThreads) {       // slices z0 - 1 .. z0 + zc, zero outside the box
            const int c = e / nx, q = e - c * nx, zz = q / HW, r = q - zz * HW, y = r / W, z = z0 - 1 + zz;
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int ci = 8 * c + k;
                v[k] = z >= 0 && z < D && ci < Cin ? in[((long long)b * Cin + ci) * S + z * HW + r] : 0.0f;
            }
            tcs_put8(xp, 16u * xrows, NT, c, (zz * hp + y + 1) * wp + (r - y * W) + 1, v);
        }
        __syncthreads();
        const uint32_t gbase = tcs_u32(gp), xbase = tcs_u32(xp);
        for (int k0 = 0; k0 < ng; k0 += 16) {
            // A: rows co, K = voxels k0 .. k0 + 15 (matrices: chunk, chunk + 1, then the upper eight voxels)
            const int ka = k0 + (lane & 7) + ((lane >> 4) & 1) * 8, ca = (lane >> 3) & 1;
            // B: K = the same voxels shifted by the tap, columns ci (matrices: lower, upper eight voxels per chunk)
            const int kb = k0 + (lane & 7) + ((lane >> 3) & 1) * 8;
            const uint32_t xr = (uint32_t)(xrow[kb] + shift);
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                uint32_t af[3][4];
#pragma unroll
                for (int p = 0; p < 3; ++p) ldsm4t(gbase + 16u * ((uint32_t)((p * MT + i) * 2 + ca) * grows + ka), af[p]);
                wg_step<NT>(acc[i], af, xbase, (uint32_t)xrows, xr, lane);
            }
        }
    }
    // partial sums [tap][co][ci] of this CTA
    float* o = part + (long long)blockIdx.x * 27 * Cout * Cin + (long long)warp * Cout * Cin;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int co = 16 * i + (lane >> 2) + 8 * (q >> 1), ci = 8 * j + 2 * (lane & 3) + (q & 1);
                if (co < Cout && ci < Cin) o[co * Cin + ci] = acc[i][j][q];
            }
}

// Output layer (one channel of g): the taps become the rows of g (im2col), and all
// of its gradient is one product over K = voxels, out[tap][ci] = sum_q g[q - tap]
// in[ci][q].  A tap per warp as above would pad the single channel to 16 rows 27
// times over (256 samples of 5 x 10 x 10, 32 channels: 84 us against 42).  (For
// the first layer the same with 27 columns per input channel lost, 118 us against
// 56: it stages 108 gathered columns per voxel.)  The warps share the K steps of
// an item (one sample's slab) and are added in warp order at the end.
// ---------------------------------------------------------------------------
constexpr int kImThreads = 256;
__host__ __device__ inline uint32_t im_smem(int HW, int zc, int mt, int nt) {
    const uint32_t rows = (uint32_t)((zc * HW + 15) & ~15);
    const uint32_t planes = 16u * 3u * rows * (uint32_t)(2 * mt + nt), red = 4u * 8u * 16u * mt * 8u * nt;
    return planes > red ? planes : red;
}
template <int NT>
__global__ void __launch_bounds__(kImThreads, 1)
k_tc_wgrad_out(int D, int H, int W, int zc, int batch, int Cin, const float* __restrict__ gsrc,
               const float* __restrict__ in, float* __restrict__ part) {
    extern __shared__ __align__(128) unsigned char tcsm[];
    constexpr int MT = 2;                                        // 27 taps in 32 rows
    const int S = D * H * W, HW = H * W, rows = (zc * HW + 15) & ~15;
    unsigned char* ap = tcsm;                                    // [piece][2 MT chunks][rows] x 16 bytes
    unsigned char* bp = ap + 16u * 3u * 2 * MT * rows;           // [piece][NT chunks][rows] x 16 bytes
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nz = (D + zc - 1) / zc, items = batch * nz;
    float acc[MT][NT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int b = it / nz, z0 = (it - b * nz) * zc, ng = (min(D, z0 + zc) - z0) * HW;
        const float* gb = gsrc + (long long)b * S;
        const float* ib = in + (long long)b * Cin * S;
        __syncthreads();                                         // the previous item's planes are read
        for (int e = tid; e < (2 * MT + NT) * rows; e += kImThreads) {
            const int c = e / rows, q = e - c * rows;
            const int pv = z0 * HW + q, z = pv / HW, r = pv - z * HW, y = r / W, x = r - y * W;
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                v[k] = 0.0f;
                if (q >= ng) continue;
                if (c < 2 * MT) {
                    const int tap = 8 * c + k, zz = z - (tap / 9 - 1), yy = y - ((tap / 3) % 3 - 1), xx = x - (tap % 3 - 1);
                    if (tap < 27 && zz >= 0 && zz < D && yy >= 0 && yy < H && xx >= 0 && xx < W) v[k] = gb[(zz * H + yy) * W + xx];
                } else {
                    const int ci = 8 * (c - 2 * MT) + k;
                    if (ci < Cin) v[k] = ib[(long long)ci * S + pv];
                }
            }
            const bool isA = c < 2 * MT;
            tcs_put8(isA ? ap : bp, 16u * rows, isA ? 2 * MT : NT, isA ? c : c - 2 * MT, q, v);
        }
        __syncthreads();
        const uint32_t abase = tcs_u32(ap), bbase = tcs_u32(bp);
        for (int k0 = 16 * warp; k0 < ng; k0 += 16 * (kImThreads / 32)) {
            const int ka = k0 + (lane & 7) + ((lane >> 4) & 1) * 8, ca = (lane >> 3) & 1;
            const uint32_t kb = (uint32_t)(k0 + (lane & 7) + ((lane >> 3) & 1) * 8);
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                uint32_t af[3][4];
#pragma unroll
                for (int p = 0; p < 3; ++p) ldsm4t(abase + 16u * ((uint32_t)((p * MT + i) * 2 + ca) * rows + ka), af[p]);
                wg_step<NT>(acc[i], af, bbase, (uint32_t)rows, kb, lane);
            }
        }
    }
    __syncthreads();
    float* red = reinterpret_cast<float*>(tcsm);                 // [warp][row][column]
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int row = 16 * i + (lane >> 2) + 8 * (q >> 1), col = 8 * j + 2 * (lane & 3) + (q & 1);
                red[(warp * 16 * MT + row) * 8 * NT + col] = acc[i][j][q];
            }
    __syncthreads();
    float* o = part + (long long)blockIdx.x * 27 * Cin;          // [tap][ci]
    for (int e = tid; e < 27 * 8 * NT; e += kImThreads) {
        const int row = e / (8 * NT), col = e - row * 8 * NT;
        float s = 0.0f;
        for (int w = 0; w < kImThreads / 32; ++w) s += red[(w * 16 * MT + row) * 8 * NT + col];
        if (col < Cin) o[row * Cin + col] = s;
    }
}

// Gradients of every parameter from the partial sums, one launch: 32 parameters
// per CTA, eight warps over the partial sums (a weight: one per CTA of its layer's
// product; a bias: one per sample), added in a fixed order.
struct TcSum { int layers; int cin[kTcMaxLayers], cout[kTcMaxLayers]; long long w_off[kTcMaxLayers], b_off[kTcMaxLayers];
               long long part[kTcMaxLayers], bpart[kTcMaxLayers]; int parts[kTcMaxLayers]; int batch; };
__global__ void __launch_bounds__(256) k_tc_sum(const __grid_constant__ TcSum a, const float* __restrict__ part,
                                                const float* __restrict__ bpart, float* __restrict__ grad) {
    int l = 0, first = 0;                                        // this CTA's layer and first parameter there
    for (;; ++l) {
        const int blocks = (27 * a.cin[l] * a.cout[l] + a.cout[l] + 31) / 32;
        if ((int)blockIdx.x < first + blocks) break;
        first += blocks;
    }
    const int ci = a.cin[l], co = a.cout[l], n = 27 * ci * co;
    const int e = ((int)blockIdx.x - first) * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
    const bool isw = e < n, live = e < n + co;
    const float* src = isw ? part + a.part[l] + e : bpart + a.bpart[l] + (e - n);
    const int cnt = !live ? 0 : isw ? a.parts[l] : a.batch;
    const long long step = isw ? n : co;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int c = w; c < cnt; c += 32)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (c + 8 * u < cnt) s[u] += src[(long long)(c + 8 * u) * step];
    __shared__ float red[8][32];
    red[w][threadIdx.x & 31] = (s[0] + s[1]) + (s[2] + s[3]);
    __syncthreads();
    if (w == 0 && live) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
        if (isw) {
            const int tap = e / (co * ci), r = e - tap * co * ci;
            grad[a.w_off[l] + (long long)r * 27 + tap] = t;
        } else {
            grad[a.b_off[l] + e - n] = t;
        }
    }
}

struct TcOffs { long long o[kTcMaxLayers]; };
// bpart[layer][b][co] = sum over the voxels of g; a warp per row, all layers in one launch.
__global__ void __launch_bounds__(256) k_tc_bias(const __grid_constant__ TcSum a, int S, const float* __restrict__ g_out,
                                                 const float* __restrict__ g, const __grid_constant__ TcOffs goff,
                                                 float* __restrict__ bpart) {
    const int l = blockIdx.y, co = a.cout[l], rows = a.batch * co;
    const float* src = l + 1 == a.layers ? g_out : g + goff.o[l];
    const int lane = threadIdx.x & 31;
    for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
        float s0 = 0.f, s1 = 0.f;
        for (int p = lane; p < S; p += 64) {
            s0 += src[(long long)r * S + p];
            if (p + 32 < S) s1 += src[(long long)r * S + p + 32];
        }
        s0 += s1;
        for (int o = 16; o > 0; o >>= 1) s0 += __shfl_down_sync(0xffffffffu, s0, o);
        if (lane == 0) bpart[a.bpart[l] + r] = s0;
    }
}

}  // namespace mrcm
