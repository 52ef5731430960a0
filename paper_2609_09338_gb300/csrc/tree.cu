// Verification of a draft tree (topk > 1): the multi-candidate form of the
// Sec. 3.1 rule over a branching chain.  At depth i the k candidates x_{i,j}
// (independent draws from the drafter's q_i; candidate 0 continues the chain)
// are tried in order against the residual r of the current node's target
// distribution p: x is accepted iff u_accept < r(x) / q_i(x), and a rejection
// replaces r by norm(max(0, r - q_i)).  Written as r = max(0, p - c q_i) / W,
// a rejection is c <- c + W, W <- sum_x max(0, p(x) - c q_i(x)) (one pass over
// the two rows), starting from c = 0, W = 1 (r = p).  An accepted chain
// candidate moves the walk one depth down; an accepted leaf, or the last
// depth, ends it with a draw from the accepted node's target row; k rejections
// end it with a draw from the last residual.  Greedy: the node's argmax is
// accepted if it is a candidate (the first such).
//
// One cluster of up to 8 blocks (512 threads each) per sequence walks its tree: block k
// takes the k-th range of the vocabulary; many sequences or short rows take fewer
// blocks each (tree_cluster).  A walk is a chain of dependent passes
// over one or two rows, so its time is the passes' latency.  One block a sequence
// pulled 1.2 MB a depth through one SM; 8 blocks pull it through as many, by bulk
// copies to shared memory, so the passes after the first (a rejection's residual
// mass, the draw) touch no global memory.  Every pass ends in one exchange of the
// warps' partials through distributed shared memory, after which all threads hold
// the same sums and take the same branch; the rows that the chain candidate leads
// to are on their way to L2 while a depth is decided.  Rows off the path are not
// waited for.  8 sequences, V 151936, float32, K 5, topk 4: 204 us with one block
// a sequence, 50 now; a depth is 7 us (rows 1.8, exponentials 3.3, exchange and
// the reduction after it 1.9).  16 blocks of 256 threads were within 5 %, 4 blocks
// 1.5 times slower.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "sizes.h"
#include "tma.cuh"

namespace osp {

namespace cg = cooperative_groups;

constexpr int TR_CS = 8;          // blocks per cluster at most (an exchange has a lane per block)
constexpr int TR_THREADS = 512;
constexpr int TR_WARPS = TR_THREADS / 32;
constexpr int TR_CH = 256;       // ids per chunk: 32 lanes x 8
constexpr int TR_U = 1;          // chunks a warp loads before using them
constexpr int TR_UG = 4;         // ... in an argmax pass
constexpr int TR_NP = 4;         // pieces a slice arrives in
constexpr size_t TREE_SMEM_CAP = 216 * 1024;
constexpr size_t TREE_SMEM_SM = 228 * 1024, TREE_SMEM_BLOCK = 6 * 1024;   // of an SM; a block's static part and the system's
constexpr float TR_LOG2E = 1.4426950408889634f;

__device__ __forceinline__ float tr_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <typename T> __device__ __forceinline__ float tr_f(T v);
template <> __device__ __forceinline__ float tr_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float tr_f<uint16_t>(uint16_t v) { return bf_to_f(v); }

// The lane's 8 logits of chunk c (ids c*256 + 8*lane ..), -inf past V.
template <typename T, bool VEC>
__device__ __forceinline__ void tr_load8(const T *row, int c, int V, float (&f)[8]) {
    const int e0 = c * TR_CH + (threadIdx.x & 31) * 8;
    if (VEC) {   // V % 8 == 0 and 16-byte rows: a vector is wholly in or out
        if (e0 < V) {
            if (sizeof(T) == 4) {
                const uint4 a = ld_stream(row + e0), b = ld_stream(row + e0 + 4);
                f[0] = __uint_as_float(a.x); f[1] = __uint_as_float(a.y);
                f[2] = __uint_as_float(a.z); f[3] = __uint_as_float(a.w);
                f[4] = __uint_as_float(b.x); f[5] = __uint_as_float(b.y);
                f[6] = __uint_as_float(b.z); f[7] = __uint_as_float(b.w);
            } else {
                unpack8(ld_stream(row + e0), f);
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = -INFINITY;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = e0 + e < V ? tr_f<T>(row[e0 + e]) : -INFINITY;
    }
}

template <typename T>
__device__ __forceinline__ float tr_at(const T *row, int x) { return tr_f<T>(row[x]); }

struct TrNorm {   // p(x) = 2^(z c2 - mp) / Sp (and q alike), c2 = log2(e) / T
    float c2, mp, isp, mq, isq;
};
// P, Q: (max, sum exp) of z / T.  A row without a finite logit has no mass.
__device__ __forceinline__ TrNorm tr_norm(float invT, MS P, MS Q) {
    const bool np = P.m == -INFINITY, nq = Q.m == -INFINITY;
    return TrNorm{invT * TR_LOG2E, np ? 0.f : P.m * TR_LOG2E, np ? 0.f : 1.f / P.s, nq ? 0.f : Q.m * TR_LOG2E,
                  nq ? 0.f : 1.f / Q.s};
}

// One block's view of the cluster and of its slice, chunks [c_lo, c_hi) of the
// vocabulary.
template <typename T>
struct TrCtx {
    cg::cluster_group cluster;
    int rank, cs, c_lo, c_hi, V, n_ex, n_fill;
    bool cached;         // the slice fits shared memory
    float *csum;         // [slice chunks]
    T *zp, *zq;          // [slice chunks][256] the current node's rows (when cached)
    float4 (*slots)[TR_CS * TR_WARPS];   // [2][cs][warps] exchange slots, used in turn
    uint64_t *full;      // [TR_NP] pieces of the slice landed
    int32_t *status;
};

// Every warp's v of every block, in (block, warp) order, through distributed
// shared memory: one cluster barrier an exchange.  The slots alternate: a slot
// is written again only after the next exchange's barrier, which every block
// reaches after it has read this one.  v is lane 0's.
template <typename T>
__device__ __forceinline__ const float4 *tr_exchange(TrCtx<T> &t, float4 v) {
    float4 *slot = t.slots[t.n_ex++ & 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    v.x = __shfl_sync(0xffffffffu, v.x, 0);
    v.y = __shfl_sync(0xffffffffu, v.y, 0);
    v.z = __shfl_sync(0xffffffffu, v.z, 0);
    v.w = __shfl_sync(0xffffffffu, v.w, 0);
    if (lane < t.cs) *t.cluster.map_shared_rank(&slot[t.rank * TR_WARPS + warp], lane) = v;
    t.cluster.sync();
    return slot;
}

// Sum of the exchanged values' x, the same in every thread of the cluster.
template <typename T>
__device__ __forceinline__ float tr_sum(const TrCtx<T> &t, const float4 *all) {
    float w = 0.f;
    for (int i = threadIdx.x & 31; i < t.cs * TR_WARPS; i += 32) w += all[i].x;
    return warp_sum(w);
}

// Piece p of the slice's chunks.
template <typename T>
__device__ __forceinline__ void tr_piece(const TrCtx<T> &t, int p, int &lo, int &hi) {
    const int n = t.c_hi - t.c_lo;
    lo = t.c_lo + n * p / TR_NP;
    hi = t.c_lo + n * (p + 1) / TR_NP;
}
__device__ __forceinline__ void tr_prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The slices of row zp (and zq when given) on their way to shared memory: bulk
// copies in TR_NP pieces where rows are 16-byte aligned, else plain loads (32
// consecutive ids each) and a block barrier.  The block has read the slices'
// last contents (a barrier before the call).
template <typename T, bool VEC>
__device__ void tr_fill(TrCtx<T> &t, const T *zp, const T *zq) {
    if (VEC) {
        if (threadIdx.x == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
#pragma unroll 1
            for (int p = 0; p < TR_NP; ++p) {
                int lo, hi;
                tr_piece(t, p, lo, hi);
                const int e0 = lo * TR_CH, e1 = min(t.V, hi * TR_CH);
                const uint32_t bytes = e1 > e0 ? (uint32_t)(e1 - e0) * sizeof(T) : 0;   // a multiple of 16 (V % 8 == 0)
                const size_t at = (size_t)(lo - t.c_lo) * TR_CH;
                mbar_arrive_expect_tx(&t.full[p], zq ? 2 * bytes : bytes);
                if (bytes) {
                    bulk_g2s(t.zp + at, zp + e0, bytes, &t.full[p]);
                    if (zq) bulk_g2s(t.zq + at, zq + e0, bytes, &t.full[p]);
                }
            }
        }
    } else {
        const int e1 = min(t.V, t.c_hi * TR_CH);
#pragma unroll 4
        for (int e = t.c_lo * TR_CH + (int)threadIdx.x; e < e1; e += TR_THREADS) {
            t.zp[e - t.c_lo * TR_CH] = zp[e];
            if (zq) t.zq[e - t.c_lo * TR_CH] = zq[e];
        }
        __syncthreads();
    }
}

// The lane's 8 logits of chunk c of the current node's row, -inf past V.
template <typename T, bool VEC>
__device__ __forceinline__ void tr_get8(const TrCtx<T> &t, const T *slice, const T *row, int c, float (&f)[8]) {
    if (t.cached) {
        const int lane = threadIdx.x & 31;
        const T *d = slice + (size_t)(c - t.c_lo) * TR_CH + lane * 8;
        if constexpr (sizeof(T) == 4) {
            const float4 a = *(const float4 *)d, b = *(const float4 *)(d + 4);
            f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
            f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
        } else {
            unpack8(*(const uint4 *)d, f);
        }
        if ((c + 1) * TR_CH > t.V) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (c * TR_CH + lane * 8 + e >= t.V) f[e] = -INFINITY;
        }
    } else {
        tr_load8<T, VEC>(row, c, t.V, f);
    }
}

// (max, sum exp) of y = z / T over row zp (and row zq when given), whose slices
// tr_fill has requested (when cached).
template <typename T, bool VEC>
__device__ void tr_stats(TrCtx<T> &t, const T *zp, const T *zq, float invT, MS &P, MS &Q) {
    const int warp = threadIdx.x >> 5;
    // maxima of the raw logits (order is kept by the positive 1/T), sums of
    // 2^((z - max) c2); four sums a row, the loads and exponentials of TR_U chunks
    // independent of one another (16 warps an SM hide little latency)
    const float c2 = invT * TR_LOG2E;
    float mp = -INFINITY, sp = 0.f, mq = -INFINITY, sq = 0.f;
    auto fold = [&](const float (&f)[TR_U][8], float &m, float &s) {
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            x[j] = fmaxf(f[0][j], f[0][j + 4]);
#pragma unroll
            for (int u = 1; u < TR_U; ++u) x[j] = fmaxf(x[j], fmaxf(f[u][j], f[u][j + 4]));
        }
        const float lm = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
        if (lm > m) {
            s = m == -INFINITY ? 0.f : s * tr_ex2((m - lm) * c2);
            m = lm;
        }
        if (m == -INFINITY) return;
        float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int u = 0; u < TR_U; ++u)
#pragma unroll
            for (int j = 0; j < 8; ++j) e[j & 3] += tr_ex2((f[u][j] - m) * c2);
        s += (e[0] + e[1]) + (e[2] + e[3]);
    };
    {
        // a warp waits for a piece when it comes to the first of its chunks there;
        // on expiry the walk goes on (every block takes part in the cluster's
        // barriers) and its result is void, which the status word says
        const bool pieces = t.cached && VEC;
        int p = -1, plo, phi = t.c_lo;
        for (int c0 = t.c_lo + warp; c0 < t.c_hi; c0 += TR_WARPS * TR_U) {
            const int last = min(t.c_hi - 1, c0 + (TR_U - 1) * TR_WARPS);
            while (pieces && last >= phi) {
                tr_piece(t, ++p, plo, phi);
                if (!mbar_wait(&t.full[p], t.n_fill & 1)) set_status(t.status, OSPREY_ERR_TIMEOUT);
            }
            float f[TR_U][8], g[TR_U][8];
#pragma unroll
            for (int u = 0; u < TR_U; ++u) {
                const int c = c0 + u * TR_WARPS;
                if (c < t.c_hi) {
                    tr_get8<T, VEC>(t, t.zp, zp, c, f[u]);
                    if (zq) tr_get8<T, VEC>(t, t.zq, zq, c, g[u]);
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) f[u][e] = g[u][e] = -INFINITY;
                }
            }
            fold(f, mp, sp);
            if (zq) fold(g, mq, sq);
        }
        // the pieces that a warp without chunks there has not waited for
        while (pieces && ++p < TR_NP)
            if (!mbar_wait(&t.full[p], t.n_fill & 1)) set_status(t.status, OSPREY_ERR_TIMEOUT);
    }
    ++t.n_fill;
    auto reduce = [&](float m, float s) {   // the warp maximum first, then each sum rescaled once
        const float M = warp_max(m);
        return MS{M * invT, warp_sum(m == -INFINITY ? 0.f : s * tr_ex2((m - M) * c2))};
    };
    P = reduce(mp, sp);
    Q = zq ? reduce(mq, sq) : MS{-INFINITY, 0.f};
    const float4 *all = tr_exchange(t, make_float4(P.m, P.s, Q.m, Q.s));
    float m1 = -INFINITY, m2 = -INFINITY;
    const int lane = threadIdx.x & 31, n = t.cs * TR_WARPS;
    for (int i = lane; i < n; i += 32) {
        m1 = fmaxf(m1, all[i].x);
        m2 = fmaxf(m2, all[i].z);
    }
    m1 = warp_max(m1);
    m2 = warp_max(m2);
    float s1 = 0.f, s2 = 0.f;
    for (int i = lane; i < n; i += 32) {
        const float4 v = all[i];
        s1 += v.x == -INFINITY ? 0.f : v.y * tr_ex2((v.x - m1) * TR_LOG2E);
        s2 += v.z == -INFINITY ? 0.f : v.w * tr_ex2((v.z - m2) * TR_LOG2E);
    }
    P = MS{m1, warp_sum(s1)};
    Q = MS{m2, warp_sum(s2)};
}

// argmax (lowest id on ties) of a row
template <typename T, bool VEC>
__device__ int tr_argmax(TrCtx<T> &t, const T *z) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, V = t.V;
    AM am{-INFINITY, 0x7fffffff};
    // Chunks past the slice: skipped by a branch in float32 (64 registers, the loads of
    // TR_UG chunks together: 256 sequences of V 151936 90 us, without it 130), loaded as
    // -inf in bf16 (40 registers, three blocks an SM: 512 of V 32000 35 us, with it 50).
    for (int c0 = t.c_lo + warp; c0 < t.c_hi; c0 += TR_WARPS * TR_UG) {
        float f[TR_UG][8];
#pragma unroll
        for (int u = 0; u < TR_UG; ++u) {
            int c = c0 + u * TR_WARPS;
            if (sizeof(T) == 4 && c >= t.c_hi) continue;
            if (sizeof(T) == 2) c = c < t.c_hi ? c : (V + TR_CH - 1) / TR_CH;   // past the row: -inf (see below)
            if (VEC) {
                tr_load8<T, VEC>(z, c, V, f[u]);
            } else {   // unaligned rows: 32 consecutive ids a load instead of a vector per lane
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int id = c * TR_CH + e * 32 + lane;
                    f[u][e] = id < V ? tr_f<T>(z[id]) : -INFINITY;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < TR_UG; ++u) {
            const int c = c0 + u * TR_WARPS;
            if (sizeof(T) == 4 && c >= t.c_hi) continue;
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (f[u][e] > am.v) am = AM{f[u][e], c * TR_CH + (VEC ? lane * 8 + e : e * 32 + lane)};
        }
    }
    am = warp_am(am);
    const float4 *all = tr_exchange(t, make_float4(am.v, __int_as_float(am.i), 0.f, 0.f));
    AM r{-INFINITY, 0x7fffffff};
    for (int i = lane; i < t.cs * TR_WARPS; i += 32) r = am_combine(r, AM{all[i].x, __float_as_int(all[i].y)});
    return warp_am(r).i;
}

// Weight of one id in a draw: the residual max(0, p - c q) (c > 0; ciq = c / Sq)
// or p.  A logit of -inf weighs 0 (2^-inf).
__device__ __forceinline__ float tr_weight(float zp, float zq, const TrNorm &n, float c, float ciq) {
    const float p = tr_ex2(fmaf(zp, n.c2, -n.mp)) * n.isp;
    return c == 0.f ? p : fmaxf(0.f, fmaf(-ciq, tr_ex2(fmaf(zq, n.c2, -n.mq)), p));
}

// The warp's sum over its chunks of tr_weight; `sums`: each chunk's sum is kept.
template <typename T, bool VEC>
__device__ float tr_warp_mass(TrCtx<T> &t, const T *zp, const T *zq, const TrNorm &n, float c, bool sums) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float ciq = c * n.isq;
    float acc = 0.f;
    for (int c0 = t.c_lo + warp; c0 < t.c_hi; c0 += TR_WARPS * TR_U) {
        float f[TR_U][8], g[TR_U][8];
#pragma unroll
        for (int u = 0; u < TR_U; ++u) {
            const int ch = c0 + u * TR_WARPS;
            if (ch < t.c_hi) {
                tr_get8<T, VEC>(t, t.zp, zp, ch, f[u]);
                if (c != 0.f) tr_get8<T, VEC>(t, t.zq, zq, ch, g[u]);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) f[u][e] = g[u][e] = -INFINITY;
            }
        }
#pragma unroll
        for (int u = 0; u < TR_U; ++u) {
            const int ch = c0 + u * TR_WARPS;
            float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < 8; ++j) e[j & 3] += tr_weight(f[u][j], g[u][j], n, c, ciq);
            float s = (e[0] + e[1]) + (e[2] + e[3]);
            if (sums) {
                s = warp_sum(s);
                if (lane == 0 && ch < t.c_hi) t.csum[ch - t.c_lo] = s;
                acc += lane == 0 ? s : 0.f;   // every lane holds the chunk's sum: count it once
            } else {
                acc += s;
            }
        }
    }
    return warp_sum(acc);
}

template <typename T, bool VEC>
__device__ float tr_mass(TrCtx<T> &t, const T *zp, const T *zq, const TrNorm &n, float c) {
    const float w = tr_warp_mass<T, VEC>(t, zp, zq, n, c, false);
    return tr_sum(t, tr_exchange(t, make_float4(w, 0.f, 0.f, 0.f)));
}

// Inverse CDF over ascending ids of tr_weight at u: a mass pass with chunk sums,
// then the block whose range holds the point finds the chunk by a scan over its
// chunk sums and the id by a warp scan, and writes the token and its flags
// (flag | 16 when rounding leaves u*S past the last sum: the last id with weight
// is taken).  The walk ends with it.
template <typename T, bool VEC>
__device__ void tr_draw(TrCtx<T> &t, const T *zp, const T *zq, const TrNorm &n, float c, float u, float *shf, int *shi,
                        int flag, int32_t *out, uint8_t *fl) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nch = t.c_hi - t.c_lo;
    const float w0 = tr_warp_mass<T, VEC>(t, zp, zq, n, c, true);
    const float4 *all = tr_exchange(t, make_float4(w0, 0.f, 0.f, 0.f));
    // block totals in vocabulary order (lane k: block k), their prefix, the owner
    float bt = 0.f;
    if (lane < t.cs)
        for (int w = 0; w < TR_WARPS; ++w) bt += all[lane * TR_WARPS + w].x;
    const float incl = warp_incl_scan(bt);
    const float S = __shfl_sync(0xffffffffu, incl, t.cs - 1);
    const float target = u * S;
    const unsigned hits = __ballot_sync(0xffffffffu, bt > 0.f && target < incl);
    const unsigned some = __ballot_sync(0xffffffffu, bt > 0.f);
    const int owner = hits ? __ffs(hits) - 1 : (some ? 31 - __clz(some) : 0);
    const float before = __shfl_sync(0xffffffffu, incl - bt, owner);
    bool past = !hits;
    if (owner != t.rank) return;
    // chunks per thread, in order
    const int per = (nch + TR_THREADS - 1) / TR_THREADS;
    const int k0 = min(nch, (int)threadIdx.x * per), k1 = min(nch, k0 + per);
    float mine_w = 0.f;
    for (int k = k0; k < k1; ++k) mine_w += t.csum[k];   // the exchange's barrier made them visible
    float tot;
    const float ex = before + block_excl_scan(mine_w, shf, &tot);
    if (threadIdx.x == 0) { shi[0] = 0x7fffffff; shi[1] = -1; }
    __syncthreads();
    if (mine_w > 0.f && target < ex + mine_w) atomicMin(&shi[0], (int)threadIdx.x);
    if (mine_w > 0.f) atomicMax(&shi[1], (int)threadIdx.x);
    __syncthreads();
    const int ct = shi[0] != 0x7fffffff ? shi[0] : (shi[1] >= 0 ? shi[1] : 0);
    past |= shi[0] == 0x7fffffff;
    __syncthreads();
    if ((int)threadIdx.x == ct) {
        float cum = ex;
        int ch = -1, lastc = k0;
        float lb = ex;
        for (int k = k0; k < k1; ++k) {
            if (t.csum[k] > 0.f) { lastc = k; lb = cum; }
            if (t.csum[k] > 0.f && target < cum + t.csum[k]) { ch = k; break; }
            cum += t.csum[k];
        }
        shi[2] = min(ch >= 0 ? ch : lastc, nch - 1);
        shf[33] = ch >= 0 ? cum : lb;
        shi[3] = ch < 0 || past;
    }
    __syncthreads();
    if (warp == 0) {
        const int ch = t.c_lo + shi[2];
        float f[8], g[8];
        tr_get8<T, VEC>(t, t.zp, zp, ch, f);
        if (c != 0.f) tr_get8<T, VEC>(t, t.zq, zq, ch, g);
        float w[8], s = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            w[e] = tr_weight(f[e], g[e], n, c, c * n.isq);
            s += w[e];
        }
        const float run = warp_incl_scan(s);
        float cum = shf[33] + run - s;
        int found = -1, lastp = -1;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            cum += w[e];
            if (w[e] > 0.f) lastp = e;
            if (found < 0 && w[e] > 0.f && target < cum) found = e;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, found >= 0);
        const unsigned pos = __ballot_sync(0xffffffffu, lastp >= 0);
        const int l = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
        if (lane == l) {
            const int e = found >= 0 ? found : (lastp >= 0 ? lastp : 0);
            *out = ch * TR_CH + l * 8 + e;
            *fl = (uint8_t)(flag | (!hit || shi[3] ? 16 : 0));
        }
    }
}

template <typename T, bool VEC, bool GREEDY>
__global__ void __launch_bounds__(TR_THREADS) tree_verify_kernel(const VerifyTreeArgs a, int slice_chunks, int cached) {
    extern __shared__ __align__(128) uint8_t dyn[];   // cached: [2][slice][256] logits; then [slice] chunk sums
    __shared__ float shf[34];
    __shared__ int shi[8];
    __shared__ float4 slots[2][TR_CS * TR_WARPS];
    __shared__ __align__(8) uint64_t full[TR_NP];
    __shared__ float s_zp[8], s_zq[8], s_u[8];
    const int K = a.K, k = a.k, V = a.V;
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), b = blockIdx.x / cs;
    const int nch = (V + TR_CH - 1) / TR_CH;
    // block 0's slice is never empty; the last ones' may be
    const int c_lo = min(nch, rank * slice_chunks);
    const size_t rows = cached ? (size_t)slice_chunks * TR_CH : 0;
    T *slice = (T *)dyn;
    TrCtx<T> t{cluster, rank, cs, c_lo, min(nch, c_lo + slice_chunks), V, 0, 0, cached != 0,
               (float *)(slice + 2 * rows), slice, slice + rows, slots, full, a.status};
    if (!GREEDY && threadIdx.x == 0) {
        for (int p = 0; p < TR_NP; ++p) mbar_init(&full[p], 1);
        mbar_fence_init();
    }
    const size_t nrow = (size_t)(1 + K * k);
    const T *tp = (const T *)a.target + (size_t)b * nrow * V;
    const T *dq = GREEDY ? nullptr : (const T *)a.draft + (size_t)b * K * V;
    const int32_t *cand = a.cand + (size_t)b * K * k;
    int32_t *out = a.out_tokens + (size_t)b * (K + 1);
    uint8_t *fl = a.flags + (size_t)b * (K + 1);
    pdl_trigger();
    __syncthreads();   // the barriers are ready
    pdl_wait();
    if (!GREEDY && t.cached) tr_fill<T, VEC>(t, tp, dq);   // the root's rows, whatever the checks say
    // candidate ids outside [0, V): the sequence is reported and skipped
    bool ok = true;
    for (int i = threadIdx.x; i < K * k; i += TR_THREADS) ok &= cand[i] >= 0 && cand[i] < V;
    ok = __syncthreads_and(ok);
    const bool lead = rank == 0 && threadIdx.x == 0;
    if (rank == 0 && threadIdx.x <= K) {
        out[threadIdx.x] = -1;
        fl[threadIdx.x] = 0;
    }
    // every block has started (its shared memory may be written), and the defaults
    // above come before what other blocks of the cluster write over them
    if (cs > 1) __threadfence();
    cluster.sync();
    if (!ok) {   // the same in every block
        if (!GREEDY && VEC && t.cached)   // the copies under way land before the block can exit
            for (int p = 0; p < TR_NP; ++p) mbar_wait(&full[p], 0);
        if (lead) {
            set_status(a.status, OSPREY_ERR_INVALID_ARG);
            a.n_accepted[b] = 0;
            a.branch[b] = -1;
        }
        return;
    }
    const float invT = GREEDY ? 1.f : 1.f / a.temperature;
    int row = 0, nacc = 0, br = -1;
    // the rows that the walk reads next if the chain candidate of depth i is
    // accepted, on their way to L2 while this depth is decided
    auto tr_next_rows = [&](int i) {
        if (!VEC || GREEDY || threadIdx.x != 0) return;
        const int e0 = t.c_lo * TR_CH, e1 = min(V, t.c_hi * TR_CH);
        if (e1 <= e0) return;
        const uint32_t bytes = (uint32_t)(e1 - e0) * sizeof(T);
        tr_prefetch_l2(tp + (size_t)(1 + i * k) * V + e0, bytes);
        if (i + 1 < K) tr_prefetch_l2(dq + (size_t)(i + 1) * V + e0, bytes);
    };
    for (int i = 0; i < K; ++i) {
        const T *zp = tp + (size_t)row * V;
        if (GREEDY) {
            const int y = tr_argmax<T, VEC>(t, zp);
            int j = -1;
            for (int jj = 0; jj < k && j < 0; ++jj)
                if (cand[i * k + jj] == y) j = jj;
            if (lead) out[i] = y;
            if (j < 0) break;
            ++nacc;
            br = j;
            row = 1 + i * k + j;
            if (j > 0 || i == K - 1) {
                const int z = tr_argmax<T, VEC>(t, tp + (size_t)row * V);
                if (lead) out[i + 1] = z;
                break;
            }
            continue;
        }
        const T *zq = dq + (size_t)i * V;
        if ((int)threadIdx.x < k) {   // the candidates' logits and uniforms, in flight with the rows
            const int x = cand[i * k + threadIdx.x];
            s_zp[threadIdx.x] = tr_at<T>(zp, x);
            s_zq[threadIdx.x] = tr_at<T>(zq, x);
            s_u[threadIdx.x] = a.u_accept[((size_t)b * K + i) * k + threadIdx.x];
        }
        MS P, Q;
        tr_stats<T, VEC>(t, zp, zq, invT, P, Q);
        tr_next_rows(i);
        const TrNorm n = tr_norm(invT, P, Q);
        float c = 0.f, W = 1.f;
        int flag = 0, acc = -1;
        for (int j = 0; j < k; ++j) {   // every thread of the cluster computes the same
            const float px = tr_ex2(fmaf(s_zp[j], n.c2, -n.mp)) * n.isp;
            const float qx = tr_ex2(fmaf(s_zq[j], n.c2, -n.mq)) * n.isq;
            const float r = fmaxf(0.f, px - c * qx) / W;
            if (s_u[j] < r / qx) {
                acc = j;
                break;
            }
            // rejected: the next residual
            c += W;
            W = tr_mass<T, VEC>(t, zp, zq, n, c);
            if (!(W > 0.f)) {   // no mass left in float32: sample p instead
                c = 0.f;
                W = 1.f;
                flag |= 8;
            }
        }
        if (acc < 0) {   // every candidate rejected: a draw from the residual
            tr_draw<T, VEC>(t, zp, zq, n, c, a.u_sample[(size_t)b * (K + 1) + i], shf, shi, flag,
                            out + i, fl + i);
            break;
        }
        if (lead) {
            out[i] = cand[i * k + acc];
            fl[i] = (uint8_t)flag;
        }
        ++nacc;
        br = acc;
        row = 1 + i * k + acc;
        if (acc > 0 || i == K - 1) {   // a leaf or the last depth: the next token from the node's row
            const T *zn = tp + (size_t)row * V;
            __syncthreads();   // the slices are read no more
            if (t.cached) tr_fill<T, VEC>(t, zn, (const T *)nullptr);
            MS Pn, Qn;
            tr_stats<T, VEC>(t, zn, (const T *)nullptr, invT, Pn, Qn);
            const TrNorm nn = tr_norm(invT, Pn, MS{-INFINITY, 0.f});
            tr_draw<T, VEC>(t, zn, (const T *)nullptr, nn, 0.f, a.u_sample[(size_t)b * (K + 1) + i + 1], shf, shi, 0,
                            out + i + 1, fl + i + 1);
            break;
        }
        __syncthreads();   // the slices and candidates are read no more
        if (t.cached) tr_fill<T, VEC>(t, tp + (size_t)row * V, dq + (size_t)(i + 1) * V);
    }
    if (lead) {
        a.n_accepted[b] = nacc;
        a.branch[b] = br;
    }
}

// What an SM and the device hold of a kernel at once, queried once per device:
// blocks per SM by registers and threads, and clusters of 8, 4, 2 and 1 blocks with
// that many blocks an SM and with one (clusters stay within a GPC).
struct TreeFit {
    std::atomic<int> per_sm, full[4], one[4];
};

// A cluster's slices of V ids: chunks a block, bytes of shared memory, and whether
// they hold two rows (else the later passes read the rows again, from L2).
struct TreeSlice {
    int chunks;
    size_t smem;
    bool cached;
};
template <typename T, bool GREEDY>
static TreeSlice tree_slice(int V, int cs) {
    const int chunks = ((V + TR_CH - 1) / TR_CH + cs - 1) / cs;
    const size_t both = (size_t)chunks * (2 * TR_CH * sizeof(T) + sizeof(float));
    const bool cached = !GREEDY && both <= TREE_SMEM_CAP;
    return TreeSlice{chunks, cached ? both : chunks * sizeof(float), cached};
}

template <typename K>
static cudaLaunchConfig_t tree_config(K, int clusters, int cs, size_t smem, cudaStream_t s, cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)clusters * cs);
    cfg.blockDim = dim3(TR_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cs;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cs > 1 ? 2 : 1;   // (a block alone is a cluster of one)
    return cfg;
}

template <typename T, bool VEC, bool GREEDY>
static cudaError_t tree_launch(const VerifyTreeArgs &a, cudaStream_t s) {
    auto *kernel = tree_verify_kernel<T, VEC, GREEDY>;
    static std::atomic<int> done[kMaxDevices];
    static TreeFit fits[kMaxDevices];
    cudaLaunchAttribute attr[2];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    TreeFit &fit = fits[dev % kMaxDevices];
    e = once_per_device(done, [&] {
        cudaError_t q = allow_smem(kernel);
        int n = 0;
        if (q == cudaSuccess) q = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, TR_THREADS, 0);
        fit.per_sm = std::max(n, 1);
        for (int i = 0; i < 3 && q == cudaSuccess; ++i) {
            cudaLaunchConfig_t cfg = tree_config(kernel, 1, TR_CS >> i, 0, nullptr, attr);
            q = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
            fit.full[i] = std::max(n, 1);
            cfg.dynamicSmemBytes = TREE_SMEM_CAP;
            if (q == cudaSuccess) q = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
            fit.one[i] = std::max(n, 1);
        }
        if (q == cudaSuccess) q = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        fit.full[3] = fit.per_sm * n;
        fit.one[3] = n;
        return q;
    });
    if (e != cudaSuccess) return e;
    TreeSlice slices[4];
    bool cached[4];
    long long at_once[4];
    for (int i = 0; i < 4; ++i) {
        slices[i] = tree_slice<T, GREEDY>(a.V, TR_CS >> i);
        const int fits = (int)(TREE_SMEM_SM / (slices[i].smem + TREE_SMEM_BLOCK));   // blocks of an SM by shared memory
        cached[i] = slices[i].cached;
        at_once[i] = fits >= (int)fit.per_sm ? (int)fit.full[i] : (int)fit.one[i] * std::max(fits, 1);
    }
    const int pick = tree_cluster(a.B, (double)a.V * sizeof(T) / 1024, GREEDY, cached, at_once);
    const int cs = TR_CS >> pick;
    const TreeSlice sl = slices[pick];
    const cudaLaunchConfig_t cfg = tree_config(kernel, a.B, cs, sl.smem, s, attr);
    e = cudaLaunchKernelEx(&cfg, kernel, a, sl.chunks, (int)sl.cached);
    count_launch();
    return e;
}

template <typename T, bool VEC>
static cudaError_t tree_launch(const VerifyTreeArgs &a, cudaStream_t s) {
    return a.temperature == 0.f ? tree_launch<T, VEC, true>(a, s) : tree_launch<T, VEC, false>(a, s);
}

cudaError_t launch_verify_tree(const VerifyTreeArgs &a, cudaStream_t s) {
    const int es = a.dtype == OSPREY_F32 ? 4 : 2;
    const bool vec = a.V % 8 == 0 && (uintptr_t)a.target % 16 == 0 &&
                     (a.draft == nullptr || (uintptr_t)a.draft % 16 == 0) && ((size_t)a.V * es) % 16 == 0;
    if (a.dtype == OSPREY_F32) return vec ? tree_launch<float, true>(a, s) : tree_launch<float, false>(a, s);
    return vec ? tree_launch<uint16_t, true>(a, s) : tree_launch<uint16_t, false>(a, s);
}

}  // namespace osp
