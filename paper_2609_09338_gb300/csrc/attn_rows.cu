// Attention of a sequence's extend rows (Sec. 4, paged serving): the new rows of
// one sequence share its cached keys, so a block takes 16 (row, head) queries of
// one KV head together and streams the key range once for all of them.
//
// The decode kernels stream the range once a row, which for 8 rows of 96
// sequences read every page 8 times from L2 and spent the CUDA cores on as many
// unpacked multiply-adds.  (Block drafting keeps them, see TcArgs::block.)  16 queries a page
// are a small matrix product: mma.sync m16n8k16 fits them (a tcgen05 tile has 128
// rows) and keeps scores and outputs in registers.  It is bound by that
// instruction's rate, about one in 9 cycles an SM here: 96 of them a page take
// 840 cycles, twice what the page takes from memory.  96 sequences, 1..8 new rows,
// 16 heads on 8 KV heads, 1024..4096 keys: 356 us a launch, row by row 592.
//
// Accuracy: q and the weights p are split into three bf16 planes (24 bits; K and V
// are bf16).  The tensor core truncates what it adds to an accumulator, so no
// chain of large terms is left to it: each 16-wide product of the first plane of q
// starts at zero and is added in float32, the other planes (2^-8, 2^-16 of it)
// chain by themselves; each page's p.V starts at zero (small planes first) and
// is added to the running output in float32.
//
// A warp takes pages warp, warp + 4, ... of the range through its own
// shared-memory stages (1-D bulk copies; one page of one head is 16 x hd
// contiguous).  The fragments are read without ldmatrix: the order of a
// product's inner dimension and of its output columns is free, so a lane takes
// the 16-byte vectors that suit it (see the two products).
#include <math.h>

#include "common.cuh"
#include "draft.cuh"
#include "internal.h"
#include "tma.cuh"

namespace osp {

constexpr int AR_W = 4;          // warps per block
constexpr int AR_T = AR_W * 32;
constexpr int AR_M = 16;         // queries per block
constexpr int AR_SPLITS = 128;   // key ranges at most

// Stages per warp: two blocks of 4 warps fit an SM.
template <int HD>
struct AttnRows {
    static constexpr int PB = 16 * HD * 2;   // bytes of one page of one head (K or V)
    static constexpr int NS = HD == 128 ? 3 : 4;
    static constexpr int RING = AR_W * NS * 2 * PB;
};

__device__ __forceinline__ void ar_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1,
                                       const float (&c)[4]) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
// bf16(x1) : bf16(x0), rounded to nearest even
__device__ __forceinline__ uint32_t ar_pack(float x0, float x1) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(x1), "f"(x0));
    return r;
}
// (x0, x1) as three packed planes
__device__ __forceinline__ void ar_split(float x0, float x1, uint32_t &p0, uint32_t &p1, uint32_t &p2) {
    p0 = ar_pack(x0, x1);
    x0 -= bf_lo(p0);
    x1 -= bf_hi(p0);
    p1 = ar_pack(x0, x1);
    x0 -= bf_lo(p1);
    x1 -= bf_hi(p1);
    p2 = ar_pack(x0, x1);
}
__device__ __forceinline__ uint32_t ar_word(const uint4 &v, int i) {
    return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

template <int HD>
__global__ void __launch_bounds__(AR_T, 2) attn_rows_kernel(const AttnArgs a, int mtiles) {
    using C = AttnRows<HD>;
    constexpr int PB = C::PB, NS = C::NS, KS = HD / 16, DPL = HD / 8;   // DPL: output dims of a lane group
    extern __shared__ __align__(128) uint8_t ring[];   // [AR_W][NS][K | V][PB], then the warps' outputs
    __shared__ __align__(8) uint64_t full[AR_W][NS];
    __shared__ float sm_m[AR_W][AR_M], sm_l[AR_W][AR_M];
    __shared__ float s_w[AR_M][AR_SPLITS], s_den[AR_M];
    const Dims &D = a.dim;
    const int split = blockIdx.x, kvh = blockIdx.y, b = blockIdx.z / mtiles, tile = blockIdx.z - b * mtiles;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lg = lane >> 2, lt = lane & 3;
    const int G = D.Hq / D.Hkv, max_new = a.map.rows_per_seq;
    pdl_trigger();   // the next projection may start streaming its weights
    // query i of the sequence: its new row i / G, head i % G of the KV head's group
    const int nn = a.map.nnew[b], nq = nn * G, i0 = tile * AR_M;   // the row map was written by the prepare kernel
    if (!a.map.valid[b] || i0 >= nq) return;   // every split's block of the tile
    const int pos0 = a.map.pos0[b];
    const int n_keys = pos0 + min(nn - 1, (i0 + AR_M - 1) / G) + 1;   // what the tile's last row sees
    const int k_begin = split * a.split_len;   // a multiple of the page size
    const int k_end = min(n_keys, k_begin + a.split_len);
    const int pg0 = k_begin / 16;
    const int npg = k_end > k_begin ? (k_end - k_begin + 15) / 16 : 0;
    const int my_pages = npg > warp ? (npg - warp + AR_W - 1) / AR_W : 0;   // pages warp + j AR_W of the range
    const int32_t *ptab = a.page_table + (size_t)b * a.max_pages + pg0;
    const size_t head_stride = (size_t)D.P * HD;
    uint8_t *wring = ring + (size_t)warp * NS * 2 * PB;
    const int my_pid = lane < my_pages ? __ldg(ptab + warp + lane * AR_W) : 0;
    auto pid_of = [&](int j) {   // warp-wide
        const int p = __shfl_sync(0xffffffffu, my_pid, j & 31);
        return j < 32 ? p : __ldg(ptab + warp + j * AR_W);
    };
    auto issue = [&](int j, int page) {   // lane 0: page j of this warp into stage j % NS
        const int st = j % NS;
        uint8_t *dst = wring + (size_t)st * 2 * PB;
        mbar_arrive_expect_tx(&full[warp][st], 2 * PB);
        bulk_g2s(dst, a.k_pages + ((size_t)page * D.Hkv + kvh) * head_stride, PB, &full[warp][st]);
        bulk_g2s(dst + PB, a.v_pages + ((size_t)page * D.Hkv + kvh) * head_stride, PB, &full[warp][st]);
    };
    const int first = min(NS, my_pages);
    int pids[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) pids[j] = pid_of(j);
    int issued = 0;
    if (lane == 0) {
        for (int st = 0; st < NS; ++st) mbar_init(&full[warp][st], 1);
        mbar_fence_init();
        // committed pages (every position below pos0) are written by no kernel of this call
#pragma unroll
        for (int j = 0; j < NS; ++j)
            if (j == issued && j < first && (pg0 + warp + j * AR_W + 1) * 16 <= pos0) issue(issued++, pids[j]);
    }
    pdl_wait();   // q and this call's K/V rows come from the QKV kernels
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < NS; ++j)
            if (j >= issued && j < first) issue(j, pids[j]);
        issued = first;
    }
    __syncwarp();

    // the lane's two queries (rows lg and lg + 8 of the tile): last key they see
    int last[2];
    uint32_t qa[3][KS][4];
    const float scale = rsqrtf((float)HD);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = i0 + lg + 8 * h, j = i / G, g = i - j * G;
        const bool on = i < nq;
        last[h] = on ? pos0 + j : -1;
        const float *qp = a.q + ((size_t)(b * max_new + (on ? j : 0)) * D.Hq + kvh * G + (on ? g : 0)) * HD;
        // the inner dimension is taken in the order that gives a lane 8 consecutive
        // dims 32 c + 8 lt of every 32: k-steps 2c and 2c + 1
#pragma unroll
        for (int c = 0; c < HD / 32; ++c) {
            const float4 x = *(const float4 *)(qp + 32 * c + 8 * lt), y = *(const float4 *)(qp + 32 * c + 8 * lt + 4);
            const float f = on ? scale : 0.f;
            ar_split(x.x * f, x.y * f, qa[0][2 * c][h], qa[1][2 * c][h], qa[2][2 * c][h]);
            ar_split(x.z * f, x.w * f, qa[0][2 * c][2 + h], qa[1][2 * c][2 + h], qa[2][2 * c][2 + h]);
            ar_split(y.x * f, y.y * f, qa[0][2 * c + 1][h], qa[1][2 * c + 1][h], qa[2][2 * c + 1][h]);
            ar_split(y.z * f, y.w * f, qa[0][2 * c + 1][2 + h], qa[1][2 * c + 1][2 + h], qa[2][2 * c + 1][2 + h]);
        }
    }
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};
    float o[DPL][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < DPL; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[j][e] = 0.f;
    int consumed = 0;
    for (int j = 0; j < my_pages; ++j) {
        const int st = j % NS;
        if (!__all_sync(0xffffffffu, mbar_wait(&full[warp][st], (uint32_t)(j / NS) & 1))) {   // warp-uniform exit
            if (lane == 0) set_status(a.status, OSPREY_ERR_TIMEOUT);
            break;
        }
        consumed = j + 1;
        const uint16_t *ks = (const uint16_t *)(wring + (size_t)st * 2 * PB), *vs = ks + 16 * HD;
        const int key0 = (pg0 + warp + j * AR_W) * 16;
        // scores of 16 queries x 16 keys: lane (lg, lt) holds keys 8 n + 2 lt, + 1 of
        // its two queries; K's fragment is key 8 n + lg, dims 32 c + 8 lt .. + 7
        float s[2][4];
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            float lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 4; ++e) s[n][e] = 0.f;
#pragma unroll
            for (int c = 0; c < HD / 32; ++c) {
                const uint4 w = *(const uint4 *)(ks + (8 * n + lg) * HD + 32 * c + 8 * lt);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t b0 = ar_word(w, 2 * h), b1 = ar_word(w, 2 * h + 1);
                    float d[4];
                    ar_mma(lo, qa[2][2 * c + h], b0, b1, lo);
                    ar_mma(lo, qa[1][2 * c + h], b0, b1, lo);
                    ar_mma(d, qa[0][2 * c + h], b0, b1, zero);
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[n][e] += d[e];
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                s[n][e] += lo[e];
                const int key = key0 + 8 * n + 2 * lt + (e & 1);
                if (key > last[e >> 1] || key >= k_end) s[n][e] = -INFINITY;
            }
        }
        float corr[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float x = fmaxf(fmaxf(s[0][2 * h], s[0][2 * h + 1]), fmaxf(s[1][2 * h], s[1][2 * h + 1]));
            x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
            x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
            const float mn = fmaxf(m[h], x);
            corr[h] = mn == -INFINITY ? 1.f : __expf(m[h] - mn);
            m[h] = mn;
            l[h] *= corr[h];
        }
        uint32_t pa[3][4];
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float x0 = s[n][2 * h], x1 = s[n][2 * h + 1];
                const float p0 = x0 == -INFINITY ? 0.f : __expf(x0 - m[h]);
                const float p1 = x1 == -INFINITY ? 0.f : __expf(x1 - m[h]);
                l[h] += p0 + p1;
                ar_split(p0, p1, pa[0][2 * n + h], pa[1][2 * n + h], pa[2][2 * n + h]);
            }
        // output += p . V: lane group lg takes dims DPL lg .. + DPL - 1, one a tile, so
        // that a lane reads whole vectors of its keys 2 lt, + 1, + 8, + 9; pairs of
        // keys are put together with byte permutes
#pragma unroll
        for (int v = 0; v < DPL / 8; ++v) {
            uint4 w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                w[k] = *(const uint4 *)(vs + (2 * lt + (k & 1) + 8 * (k >> 1)) * HD + DPL * lg + 8 * v);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int odd = 0; odd < 2; ++odd) {
                    const uint32_t sel = odd ? 0x7632u : 0x5410u;
                    const uint32_t b0 = __byte_perm(ar_word(w[0], q), ar_word(w[1], q), sel);
                    const uint32_t b1 = __byte_perm(ar_word(w[2], q), ar_word(w[3], q), sel);
                    float d[4];
                    ar_mma(d, pa[2], b0, b1, zero);
                    ar_mma(d, pa[1], b0, b1, d);
                    ar_mma(d, pa[0], b0, b1, d);
                    float (&oj)[4] = o[8 * v + 2 * q + odd];
#pragma unroll
                    for (int e = 0; e < 4; ++e) oj[e] = fmaf(oj[e], corr[e >> 1], d[e]);
                }
        }
        if (j + NS < my_pages) {   // refill the stage once every lane has read it
            const int pn = pid_of(j + NS);
            __syncwarp();
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue(j + NS, pn);
                issued = j + NS + 1;
            }
        }
    }
    // after a timed-out wait: let the copies already requested land
    if (lane == 0)
        for (int j = consumed; j < issued; ++j) mbar_wait(&full[warp][j % NS], (uint32_t)(j / NS) & 1, 200000000LL);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        l[h] += __shfl_xor_sync(0xffffffffu, l[h], 1);
        l[h] += __shfl_xor_sync(0xffffffffu, l[h], 2);
        if (lt == 0) {
            sm_m[warp][lg + 8 * h] = m[h];
            sm_l[warp][lg + 8 * h] = l[h];
        }
    }
    __syncthreads();   // every warp is done with the ring, which now takes the warps' outputs
    float *so = (float *)ring;   // [AR_W][AR_M][HD]
#pragma unroll
    for (int j = 0; j < DPL; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e)
            so[((size_t)warp * AR_M + lg + 8 * (e >> 1)) * HD + (2 * lt + (e & 1)) * DPL + j] = o[j][e];
    __syncthreads();
    const int rows = min(AR_M, nq - i0), ns = a.n_splits;
    auto part = [&](int r) {   // query r of the tile: its splits' partials (max, sum, output)
        const int j = (i0 + r) / G, g = i0 + r - j * G;
        return a.part + ((size_t)(b * max_new + j) * D.Hq + kvh * G + g) * ns * (HD + 2);
    };
    for (int idx = threadIdx.x; idx < rows * HD; idx += AR_T) {
        const int r = idx / HD, dim = idx % HD;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < AR_W; ++w) M = fmaxf(M, sm_m[w][r]);
        float num = 0.f, den = 0.f;
        if (M != -INFINITY)
#pragma unroll
            for (int w = 0; w < AR_W; ++w) {
                const float f = __expf(sm_m[w][r] - M);
                num = fmaf(f, so[((size_t)w * AR_M + r) * HD + dim], num);
                den = fmaf(f, sm_l[w][r], den);
            }
        if (ns == 1) {
            const int j = (i0 + r) / G, g = i0 + r - j * G;
            attn_store(a, b * max_new + j, (kvh * G + g) * HD + dim, num / den);
        } else {
            float *pp = part(r) + (size_t)split * (HD + 2);
            pp[2 + dim] = num;
            if (dim == 0) { pp[0] = M; pp[1] = den; }
        }
    }
    if (ns == 1 || !arrive_last(a.ticket + (size_t)blockIdx.z * D.Hkv + kvh, ns)) return;
    // the tile's last block merges the splits
    for (int r = warp; r < rows; r += AR_W) {
        const float *pp = part(r);
        float M = -INFINITY, den = 0.f;
        for (int sp = lane; sp < ns; sp += 32) M = fmaxf(M, __ldcg(pp + (size_t)sp * (HD + 2)));
        M = warp_max(M);
        for (int sp = lane; sp < ns; sp += 32) {
            const float ms = __ldcg(pp + (size_t)sp * (HD + 2));
            const float f = ms == -INFINITY ? 0.f : __expf(ms - M);
            den = fmaf(f, __ldcg(pp + (size_t)sp * (HD + 2) + 1), den);
            s_w[r][sp] = f;
        }
        den = warp_sum(den);
        if (lane == 0) s_den[r] = den;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < rows * HD; idx += AR_T) {
        const int r = idx / HD, dim = idx % HD, j = (i0 + r) / G, g = i0 + r - j * G;
        const float *pp = part(r) + 2 + dim;
        float num = 0.f;
#pragma unroll 8
        for (int sp = 0; sp < ns; ++sp) num = fmaf(s_w[r][sp], __ldcg(pp + (size_t)sp * (HD + 2)), num);
        attn_store(a, b * max_new + j, (kvh * G + g) * HD + dim, num / s_den[r]);
    }
}

int attn_rows_tiles(const Dims &D, int max_new) { return (max_new * (D.Hq / D.Hkv) + AR_M - 1) / AR_M; }

template <int HD>
static cudaError_t launch_attn_rows_t(const AttnArgs &a, int B, int mtiles, cudaStream_t s) {
    static std::atomic<int> done[kMaxDevices];   // the ring's dynamic shared memory, opted into once per device
    cudaError_t e = once_per_device(done, [] {
        return cudaFuncSetAttribute(attn_rows_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnRows<HD>::RING);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.n_splits, a.dim.Hkv, B * mtiles);
    cfg.blockDim = dim3(AR_T);
    cfg.dynamicSmemBytes = AttnRows<HD>::RING;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, attn_rows_kernel<HD>, a, mtiles);
}

cudaError_t launch_attn_rows(const AttnArgs &a, int B, int mtiles, cudaStream_t s) {
    const cudaError_t e = a.dim.hd == 128 ? launch_attn_rows_t<128>(a, B, mtiles, s) : launch_attn_rows_t<64>(a, B, mtiles, s);
    count_launch();
    return e;
}

}  // namespace osp
