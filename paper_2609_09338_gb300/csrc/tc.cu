// Batched-row draft step on tcgen05 tensor cores: streamed swap-AB GEMMs for
// the projections of Sec. 3.3 (Eq. 1-3, MLP, LM head), operand preparation,
// RoPE + paged K/V write, and per-row sampling of the draft token (Sec. 3.1).
//
// tc_kernel: persistent, two CTAs per SM (one for large calls), 6 warps.
//   warp 0     issues 2-D TMA copies of one 128-row weight tile and the
//              activation planes per 64-wide k-block into
//              an nst-slot shared-memory ring (128-byte swizzle);
//   warp 1     issues tcgen05.mma (M 128, N npad, K 16, bf16 in, float32
//              accumulate in TMEM) per k-block and plane, then commits the
//              k-block to the slot's "empty" barrier and each accumulation
//              segment to its accumulator's "full" barrier;
//   warps 2-5  read the accumulator (tcgen05.ld, TMEM lane group = warp % 4)
//              and run the epilogue while the next segment accumulates into
//              the other TMEM buffer.
// What bounds it: in the decode shapes the weights' way from HBM (the LM head of 64
// rows, 410 MB: 77 us, 5.3 TB/s); with more rows shared memory, from which an MMA
// reads its weights (measured 44 cycles an MMA of 64 rows), and the ring's depth.
// Every wait is bounded; on expiry the CTA records OSPREY_ERR_TIMEOUT, stops
// issuing, lets its copies and MMAs land and frees its TMEM.
#include <cooperative_groups.h>
#include <cudaTypedefs.h>
#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"
#include "tma.cuh"

namespace osp {

namespace cg = cooperative_groups;

constexpr int TC_THREADS = 192;
constexpr int TC_ABYTES = 128 * 128;    // weight tile: 128 rows x 64 bf16
constexpr int TC_MAXST = 8;
// Two CTAs per SM are two TMA producers, MMA chains and epilogues; one has all of
// TMEM and shared memory, and tiles of up to TC_BIG_ROWS rows (tc_tiles).  An MMA
// reads its 4 KB of weights from shared memory however many rows it multiplies (32
// cycles; 16 rows more take 4), so 128 rows at once cost two thirds of twice 64.
// Two CTAs, the system's share and the static part fit 228 KB: 100 KB left the
// third stage of 48 rows and the fifth of 16 out (16 sequences, 2 layers of d
// 2048: 1992 us a call, with it 1970).
__host__ __device__ constexpr size_t tc_smem_cap(int bps) { return (size_t)(bps == 1 ? 225 : 112) * 1024; }
__host__ __device__ constexpr uint32_t tc_tmem_cols(int bps) { return 512 / bps; }   // of one CTA
#ifndef OSP_TC_SEGKB
#define OSP_TC_SEGKB 8   // k-blocks (64 wide) per accumulation segment
#endif
// Accuracy of the accumulators.  A tensor-core accumulator drops the bits below
// its last place at every step instead of rounding to nearest, so its error
// grows with the steps that add to a large value.  The planes after the first,
// 2^-8 and 2^-16 of it, therefore have an accumulator of their own, and calls of
// more rows than a tile, whose rows the CUDA-core GEMV sums in float32, take
// segments of 2 k-blocks: 8 steps at full size instead of 96.  Measured
// against float64 on 96 sequences, d 1024 (logits, cached bf16 K values that
// round otherwise; us a call): 8 k-blocks, one accumulator 1.9e-6, 1160, 4250;
// 2 k-blocks, one accumulator 4.9e-7, 370, 5140; 4 k-blocks, two 2.8e-7, 220,
// 3780; 2 k-blocks, two 1.7e-7, 170, 4020; the GEMV 1.6e-7, 220, 34500.
// The LM head of such a batch takes segments of 1: logits 1.5e-7 off instead of
// 1.7e-7 (the GEMV's 1.6e-7), for 3100 us a call instead of 2864.  What is left is
// a bias of the leading logit, of one sign in every step: -2.2e-6 at 46 (segments
// of 2: -5.5e-6), half a unit in the last place, where the GEMV has none; rms 4.3e-6
// against 2.7e-6.
// Block drafting keeps one accumulator, segments of 8 and the LM head's two planes
// at every number of rows (TcArgs::block): 2.4e-5 at d 4096.
#ifndef OSP_TC_SEGKB_FINE
#define OSP_TC_SEGKB_FINE 2
#endif
#ifndef OSP_TC_SEGKB_LM
#define OSP_TC_SEGKB_LM 1   // ... of its LM head
#endif
#ifndef OSP_TC_LM_NA
#define OSP_TC_LM_NA 2   // LM head: weight tiles per stage that share one operand stage
#endif

// ---------------------------------------------------------------- tcgen05 PTX
__device__ __forceinline__ void tma_2d(void *dst, const CUtensorMap *m, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(m), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
// Shared-memory matrix descriptor: K-major tile, rows 128 bytes apart inside
// 8-row (1024-byte) swizzle atoms.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;              // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset: one 8-row atom
    d |= (uint64_t)1 << 46;              // descriptor version
    d |= (uint64_t)2 << 61;              // 128-byte swizzle
    return d;
}
// Instruction descriptor, kind::f16: bf16 A and B (K-major), float32 D.
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"(acc)
                 : "memory");
}
// One lane of a converged warp.  A role's loop runs under this predicate rather
// than a test of the lane's number: the compiler then knows that a single thread
// issues, and keeps descriptors and addresses in uniform registers.
__device__ __forceinline__ bool tc_elect() {
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void tc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
        "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
        "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
        : "memory");
}
__device__ __forceinline__ void tc_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Keeps the uses of a tcgen05.ld's registers after the wait before this call.
__device__ __forceinline__ void tc_ld_tie(float (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j) asm volatile("" : "+f"(v[j]));
}

// x ~= q0 + q1 + q2 with q_i = bf16(x - q0 - ... - q_{i-1}): 8 significant bits
// per plane, so three planes carry a float32 value's 24 (up to the last rounding).
__device__ __forceinline__ void tc_split(float x, uint16_t (&q)[TC_PLANES]) {
    float r = x;
#pragma unroll
    for (int i = 0; i < TC_PLANES; ++i) {
        q[i] = f_to_bf(r);
        r -= bf_to_f(q[i]);
    }
}

// Merges two (argmax logit a with its id i, sum s of exp((z - a) / T)) pairs
// into the first: the larger logit wins (the lower id on ties) and the
// other's sum is rescaled to it.
__device__ __forceinline__ void lm_combine(float &a1, int &i1, float &s1, float a2, int i2, float s2, float invT) {
    const bool two = a2 > a1 || (a2 == a1 && i2 < i1);
    const float aw = two ? a2 : a1, al = two ? a1 : a2;
    const float sw = two ? s2 : s1, sl = two ? s1 : s2;
    const float f = al == -INFINITY ? 0.f : __expf((al - aw) * invT);
    a1 = aw;
    i1 = two ? i2 : i1;
    s1 = sw + sl * f;
}

// 2^x on the special-function unit (PTX ex2.approx, flush-to-zero)
__device__ __forceinline__ float lm_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---------------------------------------------------------------- GEMM kernel
// NA weight tiles (NA x 128 output features) share each stage's operand
// planes: one work item is NA adjacent tiles, accumulated side by side in TMEM.
// Output features [0, nout_a) come from the weights of map wa, the rest from
// wb (row f - nout_a): the SwiGLU gate and up projections run as one GEMM.
// a.pair CTAs next to one another take adjacent row tiles of the same features and
// k-range at the same time: the second one's weight tiles come from L2.
// BPS: CTAs per SM.
template <int EPI, int NA, int BPS>
__global__ void __launch_bounds__(TC_THREADS, BPS)
    tc_kernel(const __grid_constant__ CUtensorMap wa, const __grid_constant__ CUtensorMap wb,
              const __grid_constant__ CUtensorMap xm, const TcArgs a, int nst) {
    extern __shared__ uint8_t raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[TC_MAXST], empty[TC_MAXST], accf[2], acce[2], sepe, fin;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // work item of a pair = (NA output tiles of 128 features, a.pair row tiles,
    // k-range), the k-range fastest; items of a pair are contiguous
    const int segkb = a.segkb;
    const int pair = a.pair, nrg = a.nrt / pair, per_ft = nrg * a.nsplit;   // items of one feature tile
    const int n_items = (a.nout + 128 * NA - 1) / (128 * NA) * per_ft;
    const int rank = blockIdx.x % pair, at = blockIdx.x / pair, of = gridDim.x / pair;
    const int i0 = (int)((long long)n_items * at / of);
    const int i1 = (int)((long long)n_items * (at + 1) / of);
    const int nloc = i1 - i0, nkb = a.K / 64, npad = a.npad;
    auto krange = [&](int item, int &lo, int &hi) {
        const int sp = item % a.nsplit;
        lo = sp * a.kbps;
        hi = min(nkb, lo + a.kbps);
    };
    const uint32_t bbytes = (uint32_t)a.planes * npad * 128;
    const uint32_t stage = NA * TC_ABYTES + bbytes;
    // TMEM: two segment buffers, and with `sep` one accumulator of the planes
    // after the first over the item's whole k-range (they are 2^-8 and 2^-16 of
    // the first plane, so what their accumulator drops does not matter)
    const uint32_t acc_cols = NA * npad;
    const bool sep = NA == 1 && a.sep;
    // an item of several segments is finished from columns of its own where they
    // fit (tiles of up to 64 rows), so that its last segment's buffer is free at once
    const bool own = NA == 1 && a.kbps > a.segkb && 4 * acc_cols <= tc_tmem_cols(BPS);
    // the LM head's two weight tiles: an accumulator of the small planes beside each
    // buffer where they fit, up to 32 rows (16 rows, d 2048: logits 3.3e-6 off the
    // float64 ones instead of 5.1e-6, for 0.7 % of a call)
    const bool duo = NA > 1 && a.sep && 4 * acc_cols <= tc_tmem_cols(BPS);
    uint32_t ncols = 32;
    while (ncols < (own || duo ? 4 : sep ? 3 : 2) * acc_cols) ncols <<= 1;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 32) {
        for (int i = 0; i < nst; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&accf[i], 1);
            mbar_init(&acce[i], 4);
        }
        mbar_init(&sepe, 4);
        mbar_init(&fin, 1);
        s_abort = 0;
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    pdl_trigger();
    // the activation planes and the residual come from earlier kernels; the
    // producer first requests the weight tiles of the ring's first stages,
    // which do not, and waits after that
    if (warp != 0) pdl_wait();

    if (warp == 0) {
        if (tc_elect()) {
            auto weights = [&](uint8_t *st, int y, int kb, uint64_t *bar) {
#pragma unroll
                for (int t = 0; t < NA; ++t) {
                    const int f = y + 128 * t;   // tiles never straddle nout_a (a multiple of 128)
                    tma_2d(st + t * TC_ABYTES, f < a.nout_a ? &wa : &wb, kb * 64, f < a.nout_a ? f : f - a.nout_a, bar);
                }
            };
            int npre = 0;   // stages whose weights were requested before the wait
            for (int it = 0; it < nloc && npre < nst; ++it) {
                const int y = (i0 + it) / per_ft * 128 * NA;
                int klo, khi;
                krange(i0 + it, klo, khi);
                for (int kb = klo; kb < khi && npre < nst; ++kb, ++npre) {
                    mbar_expect_tx(&full[npre], NA * TC_ABYTES);
                    weights(sm + (size_t)npre * stage, y, kb, &full[npre]);
                }
            }
            pdl_wait();
            // slot and use of the ring advance by increments: a division by the runtime
            // number of stages, twice a k-block, took longer than its MMAs
            int g = 0, s = 0;          // k-block of the CTA, its slot
            uint32_t ph = 1;           // parity of the slot's previous use
            bool stop = false;
            for (int it = 0; it < nloc && !stop; ++it) {
                const int y = (i0 + it) / per_ft * 128 * NA;
                const int row0 = ((i0 + it) / a.nsplit % nrg * pair + rank) * npad;   // of the operand planes
                int klo, khi;
                krange(i0 + it, klo, khi);
                for (int kb = klo; kb < khi; ++kb, ++g, ++s) {
                    if (s == nst) {
                        s = 0;
                        ph ^= 1;
                    }
                    if (g >= nst && !mbar_wait(&empty[s], ph)) {
                        set_status(a.status, OSPREY_ERR_TIMEOUT);
                        atomicExch(&s_abort, 1);
                        stop = true;
                        break;
                    }
                    if (*(volatile int *)&s_abort) { stop = true; break; }
                    uint8_t *st = sm + (size_t)s * stage;
                    if (g < npre) {
                        mbar_arrive_expect_tx(&full[s], bbytes);
                    } else {
                        mbar_arrive_expect_tx(&full[s], stage);
                        weights(st, y, kb, &full[s]);
                    }
                    for (int p = 0; p < a.planes; ++p)
                        tma_2d(st + NA * TC_ABYTES + (size_t)p * npad * 128, &xm, kb * 64, p * a.prows + a.prow0 + row0,
                               &full[s]);
                }
            }
            if (stop) {   // let the copies this thread issued land before the CTA can exit
                // stages whose weights were requested early but never armed: arrive, so
                // that their phase completes when the weights land
                for (int q = g; q < npre; ++q) mbar_arrive(&full[q]);
                const int end = g > npre ? g : npre;
                for (int q = end - nst > 0 ? end - nst : 0; q < end; ++q)
                    mbar_wait(&full[q % nst], (uint32_t)(q / nst) & 1, 200000000LL);
            }
        }
    } else if (warp == 1) {
        if (tc_elect()) {
            // one accumulation unit = one segment of one tile, into buffer u & 1
            const uint32_t idesc = tc_idesc(128, npad), pstep = (uint32_t)npad * 128 >> 4;   // descriptor units a plane
            int u = 0, s = 0;          // accumulation unit, ring slot
            uint32_t ph = 0;           // parity of the slot's current use
            bool stop = false;
            for (int it = 0; it < nloc && !stop; ++it) {
                int klo, khi;
                krange(i0 + it, klo, khi);
                const int nseg = (khi - klo + segkb - 1) / segkb;
                for (int sg = 0; sg < nseg && !stop; ++sg, ++u) {
                    const int buf = u & 1;
                    if (u >= 2 && !mbar_wait(&acce[buf], (uint32_t)((u >> 1) - 1) & 1)) {
                        set_status(a.status, OSPREY_ERR_TIMEOUT);
                        atomicExch(&s_abort, 1);
                        stop = true;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d0 = tmem + (uint32_t)buf * acc_cols;
                    const int kb0 = klo + sg * segkb, kb1 = min(khi, kb0 + segkb);
                    for (int kb = kb0; kb < kb1; ++kb, ++s) {
                        if (s == nst) {
                            s = 0;
                            ph ^= 1;
                        }
                        if (!mbar_wait(&full[s], ph) || *(volatile int *)&s_abort) {
                            set_status(a.status, OSPREY_ERR_TIMEOUT);
                            atomicExch(&s_abort, 1);
                            stop = true;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t st = smem_u32(sm + (size_t)s * stage);
                        const uint64_t da = tc_desc(st), db0 = tc_desc(st + NA * TC_ABYTES);
                        auto step = [&](int p, int kk, uint32_t d, uint32_t acc) {
                            const uint64_t db = db0 + (uint64_t)(p * pstep) + 2 * kk;
#pragma unroll
                            for (int t = 0; t < NA; ++t)
                                tc_mma(d + (uint32_t)(t * npad), da + t * (TC_ABYTES >> 4) + 2 * kk, db, idesc, acc);
                        };
                        if (sep) {
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) step(0, kk, d0, (kb != kb0) || kk);
                            // the item's first small-plane step overwrites that accumulator: the
                            // epilogue has to have read the previous item's
                            if (kb == klo && it > 0 && !mbar_wait(&sepe, (uint32_t)(it - 1) & 1)) {
                                set_status(a.status, OSPREY_ERR_TIMEOUT);
                                atomicExch(&s_abort, 1);
                                stop = true;
                                break;
                            }
                            for (int p = 1; p < a.planes; ++p)
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk)
                                    step(p, kk, tmem + 2u * acc_cols, (kb != klo) || kk || p > 1);
                        } else if (a.block) {
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                for (int p = 0; p < a.planes; ++p) step(p, kk, d0, (kb != kb0) || kk || p);
                        } else {
                            // plane by plane (planes inside a k-step made the calls 1.5 % slower), the
                            // small ones first, while the accumulator is small
                            for (int p = a.planes - 1; p >= 0; --p) {
                                const uint32_t d = duo && p > 0 ? d0 + 2u * acc_cols : d0;
                                const bool first = kb == kb0 && (p == a.planes - 1 || (duo && p == 0));
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk) step(p, kk, d, !first || kk);
                            }
                        }
                        tc_commit(&empty[s]);
                    }
                    if (!stop) tc_commit(&accf[buf]);
                }
            }
            tc_commit(&fin);
            mbar_wait(&fin, 0, 400000000LL);   // every MMA of this CTA has completed
        }
    } else {
        // epilogue: TMEM lanes (warp % 4) * 32 .. + 31 hold output features m.
        const int lg = (warp & 3) * 32;
        const int m = lg + lane;
        const uint32_t lanes = tmem + ((uint32_t)lg << 16);
        int u = 0;
        bool stop = false;
        int ft = 0, sp = 0, col0 = 0, row0 = 0;
        // the finished sums v of rows row0 + c0 .. + 15, feature col0 + 128 tile
        auto finish = [&](int tile, int c0, float (&v)[16]) {
            const int col = col0 + 128 * tile;
            const bool colok = col < a.nout;
            if constexpr (EPI == TC_LM) {
                // per row: (argmax z, sum exp((z - max z) / T)) over this warp's 32 ids,
                // for the 16 rows c0.. at once: the maximum by a warp reduction, its
                // first lane by a ballot, then the sums by a butterfly that halves the
                // rows a lane carries each round (it keeps one half and receives the
                // partner's share of it), so that lane l ends with row l / 2.  About 220
                // instructions a chunk, independent across rows; merging (max, sum, id)
                // triples through the butterfly took 500 in a chain, 2.8 us a chunk
                const int sub = (int)(((long long)ft * 128 * NA + 128 * tile + lg) / TC_LM_GROUP);
                const float c2 = a.lm_invT * 1.4426950408889634f;
                float e[16], mine = -INFINITY;
                int first = -1;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (a.y && colok && row0 + c0 + j < a.R) a.y[(size_t)(row0 + c0 + j) * a.ldy + col] = v[j];
                    const float z = colok ? v[j] : -INFINITY;
                    float mx;
                    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(mx) : "f"(z));
                    const unsigned at = __ballot_sync(0xffffffffu, z == mx);
                    e[j] = mx == -INFINITY ? 0.f : lm_ex2((z - mx) * c2);
                    if ((lane >> 1) == j) {
                        mine = mx;
                        first = __ffs(at) - 1;
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int off = 16 >> r, w = 8 >> r;
                    const bool up = lane & off;
#pragma unroll
                    for (int i = 0; i < w; ++i) {
                        const float got = __shfl_xor_sync(0xffffffffu, up ? e[i] : e[i + w], off);
                        e[i] = (up ? e[i + w] : e[i]) + got;
                    }
                }
                e[0] += __shfl_xor_sync(0xffffffffu, e[0], 1);
                const int n = row0 + c0 + (lane >> 1);
                if (!(lane & 1) && n < a.R && sub < a.lm_nsub)
                    a.lm_part[(size_t)n * a.lm_nsub + sub] =
                        make_float4(mine * a.lm_invT, e[0], mine,
                                    __int_as_float(mine == -INFINITY ? 0x7fffffff : col - lane + first));
            } else if constexpr (EPI == TC_LM_BLOCK) {
                // the same partials, as (max, id, sum) triples merged through the butterfly:
                // the order that block drafting keeps (120 rows, d 4096: 361 us a launch; as above 292)
                const int sub = (int)(((long long)ft * 128 * NA + 128 * tile + lg) / TC_LM_GROUP);
                float av[16], sv[16];
                int ai[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    av[j] = colok ? v[j] : -INFINITY;
                    ai[j] = colok ? col : 0x7fffffff;
                    sv[j] = colok ? 1.f : 0.f;
                    if (a.y && colok && row0 + c0 + j < a.R) a.y[(size_t)(row0 + c0 + j) * a.ldy + col] = v[j];
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int off = 16 >> r, w = 8 >> r;
                    const bool up = lane & off;
#pragma unroll
                    for (int i = 0; i < w; ++i) {
                        const float ra = __shfl_xor_sync(0xffffffffu, up ? av[i] : av[i + w], off);
                        const int ri = __shfl_xor_sync(0xffffffffu, up ? ai[i] : ai[i + w], off);
                        const float rs = __shfl_xor_sync(0xffffffffu, up ? sv[i] : sv[i + w], off);
                        float ka = up ? av[i + w] : av[i], ks = up ? sv[i + w] : sv[i];
                        int ki = up ? ai[i + w] : ai[i];
                        lm_combine(ka, ki, ks, ra, ri, rs, a.lm_invT);
                        av[i] = ka;
                        ai[i] = ki;
                        sv[i] = ks;
                    }
                }
                const float ra = __shfl_xor_sync(0xffffffffu, av[0], 1);
                const int ri = __shfl_xor_sync(0xffffffffu, ai[0], 1);
                const float rs = __shfl_xor_sync(0xffffffffu, sv[0], 1);
                lm_combine(av[0], ai[0], sv[0], ra, ri, rs, a.lm_invT);
                const int n = row0 + c0 + (lane >> 1);
                if (!(lane & 1) && n < a.R && sub < a.lm_nsub)
                    a.lm_part[(size_t)n * a.lm_nsub + sub] =
                        make_float4(av[0] * a.lm_invT, sv[0], av[0], __int_as_float(ai[0]));
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int n = row0 + c0 + j;
                    if (n >= a.R || !colok) continue;
                    if (a.nsplit > 1 || EPI == TC_GLU) {   // partial of this k-range; tc_reduce applies the epilogue
                        a.part[((size_t)sp * a.R + n) * a.nout + col] = v[j];
                    } else if (EPI == TC_STORE) {
                        a.y[(size_t)n * a.ldy + col] = v[j];
                    } else if (EPI == TC_RESID) {
                        a.x[(size_t)n * a.ldy + col] += v[j];
                    }
                }
            }
        };
        for (int it = 0; it < nloc && !stop; ++it) {
            ft = (i0 + it) / per_ft;
            sp = (i0 + it) % a.nsplit;
            col0 = ft * 128 * NA + m;
            row0 = ((i0 + it) / a.nsplit % nrg * pair + rank) * npad;
            int klo, khi;
            krange(i0 + it, klo, khi);
            const int nseg = (khi - klo + segkb - 1) / segkb;
            auto wait_acc = [&]() {
                if (mbar_wait(&accf[u & 1], (uint32_t)(u >> 1) & 1) && !*(volatile int *)&s_abort) {
                    tc_fence_after();
                    return true;
                }
                set_status(a.status, OSPREY_ERR_TIMEOUT);
                atomicExch(&s_abort, 1);
                stop = true;
                return false;
            };
            auto release = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce[u & 1]);
            };
            if constexpr (NA == 1) {
                // several segments: the running total is kept in registers, each segment
                // added to it in float32 and its buffer freed at once, and is put back
                // into TMEM, from which the loop below finishes it
                // (a loop over chunks in TMEM: unrolled over registers, its code is five
                // times as long, which cost each short launch 5 us of instruction fetches)
                if (nseg > 1) {
                    constexpr int NCH = (BPS == 1 ? TC_BIG_ROWS : TC_TILE_ROWS) / 16;
                    const int nch = npad / 16;
                    float tot[NCH][16];
                    auto add = [&](uint32_t t0) {   // two chunks' loads in flight at a time
#pragma unroll
                        for (int c = 0; c < NCH; c += 2) {
                            float v[2][16];
                            if (c < nch) tc_ld16(t0 + 16u * c, v[0]);
                            if (c + 1 < NCH && c + 1 < nch) tc_ld16(t0 + 16u * (c + 1), v[1]);
                            tc_ld_wait();
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                if (c + i < NCH && c + i < nch) {
                                    tc_ld_tie(v[i]);
#pragma unroll
                                    for (int j = 0; j < 16; ++j) tot[c + i][j] += v[i][j];
                                }
                        }
                    };
#pragma unroll
                    for (int c = 0; c < NCH; ++c)
#pragma unroll
                        for (int j = 0; j < 16; ++j) tot[c][j] = 0.f;
                    for (int sg = 0; sg < nseg; ++sg) {
                        if (!wait_acc()) break;
                        add(lanes + (uint32_t)(u & 1) * acc_cols);
                        if (sg < nseg - 1) {
                            release();
                            ++u;
                        }
                    }
                    if (stop) break;
                    if (sep) {
                        add(lanes + 2u * acc_cols);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sepe);
                    }
                    if (own) release();
#pragma unroll
                    for (int c = 0; c < NCH; ++c)
                        if (c < nch) tc_st16(lanes + (own ? 3u : (uint32_t)(u & 1)) * acc_cols + 16u * c, tot[c]);
                    tc_st_wait();
                } else if (!wait_acc()) {
                    break;
                }
            } else if (!wait_acc()) {   // one segment an item
                break;
            }
            const bool freed = own && nseg > 1;
            const uint32_t t0 = lanes + (freed ? 3u : (uint32_t)(u & 1)) * acc_cols;
            for (int cc = 0; cc < NA * npad; cc += 16) {
                // accumulator columns [t npad, (t + 1) npad) hold tile t's rows
                const int tile = cc / npad;
                float v[16];
                tc_ld16(t0 + (uint32_t)cc, v);
                if ((sep && nseg == 1) || duo) {
                    float w[16];
                    tc_ld16((duo ? t0 : lanes) + 2u * acc_cols + (uint32_t)cc, w);
                    tc_ld_wait();
                    tc_ld_tie(v);
                    tc_ld_tie(w);
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] += w[j];
                } else {
                    tc_ld_wait();
                    tc_ld_tie(v);
                }
                finish(tile, cc - tile * npad, v);
            }
            if (!freed) release();
            if (sep && nseg == 1 && lane == 0) mbar_arrive(&sepe);   // (one segment: after release()'s warp barrier)
            ++u;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// ---------------------------------------------------------------- split-K reduction
// out[n][col] = sum over the k-ranges (in order) of the partials, then the
// GEMM's epilogue.  TC_GLU: gate = output col, up = output nout_a + col, and
// the planes of h = silu(gate) * up go to h [TC_PLANES][h_rows][nout_a].
template <int EPI>
__global__ void __launch_bounds__(256) tc_reduce_kernel(const TcArgs a) {
    pdl_trigger();
    pdl_wait();
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int w = EPI == TC_GLU ? a.nout_a : a.nout;
    if (idx >= (long long)a.R * w) return;
    const int n = (int)(idx / w), col = (int)(idx % w);
    float v = 0.f;
    for (int sp = 0; sp < a.nsplit; ++sp) v += __ldcg(a.part + ((size_t)sp * a.R + n) * a.nout + col);
    if (EPI == TC_STORE) {
        a.y[(size_t)n * a.ldy + col] = v;
    } else if (EPI == TC_RESID) {
        a.x[(size_t)n * a.ldy + col] += v;
    } else {
        float u = 0.f;
        for (int sp = 0; sp < a.nsplit; ++sp) u += __ldcg(a.part + ((size_t)sp * a.R + n) * a.nout + w + col);
        const float h = v / (1.f + expf(-v)) * u;
        uint16_t q[TC_PLANES];
        tc_split(h, q);
#pragma unroll
        for (int i = 0; i < TC_PLANES; ++i) a.h[((size_t)i * a.h_rows + n) * w + col] = q[i];
    }
}

// TC_RESID reduction with the next operand's planes: a cluster of RP_CS blocks
// per row n, each summing the partials (in range order) of its share of the
// columns into x[n]; the blocks' sums of squares are exchanged through
// distributed shared memory, then each writes the RMS-normalised planes of its
// columns.
constexpr int RP_CS = 8;     // blocks per row (one cluster)
constexpr int RP_VPT = 4;    // columns per thread at most (nout <= RP_CS * 256 * RP_VPT)
__device__ __forceinline__ void rp_cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void rp_cluster_arrive_release() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void rp_cluster_wait_acquire() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __launch_bounds__(256) tc_resid_planes_kernel(const TcArgs a) {
    __shared__ float red[8];
    __shared__ float css[RP_CS];   // every block's sum of squares, pushed by its owner
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), n = blockIdx.y, t = threadIdx.x;
    rp_cluster_arrive_relaxed();   // started: the cluster may write this block's shared memory
    pdl_trigger();
    pdl_wait();
    int prow = -1;
    bool act = false;
    if (a.pl_map == 0) {
        const int b = n / a.pl_rows_per_seq, j = n - b * a.pl_rows_per_seq;
        act = a.pl_valid[b] && (a.pl_rows_per_seq == 1 || j < a.pl_nnew[b]);
        prow = n;
    } else {
        const int b = n / a.pl_max_new, j = n - b * a.pl_max_new;
        if (a.pl_valid[b] ? j == a.pl_nnew[b] - 1 : j == 0) {
            prow = b;
            act = a.pl_valid[b] != 0;
        }
    }
    const int per = (a.nout + RP_CS - 1) / RP_CS;
    const int c0 = rank * per, c1 = min(a.nout, c0 + per);
    float xv[RP_VPT];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < RP_VPT; ++i) {
        const int col = c0 + t + 256 * i;
        xv[i] = 0.f;
        if (col >= c1) continue;
        float v = 0.f;
        for (int sp = 0; sp < a.nsplit; ++sp) v += __ldcg(a.part + ((size_t)sp * a.R + n) * a.nout + col);
        const float xn = a.x[(size_t)n * a.ldy + col] + v;
        a.x[(size_t)n * a.ldy + col] = xn;
        xv[i] = xn;
        ss = fmaf(xn, xn, ss);
    }
    if (prow < 0) return;   // the whole cluster (same row) leaves here
    ss = warp_sum(ss);
    if ((t & 31) == 0) red[t >> 5] = ss;
    __syncthreads();
    rp_cluster_wait_acquire();   // every block of the cluster has started
    if (t == 0) {
        float tot = 0.f;
        for (int w = 0; w < 8; ++w) tot += red[w];
        for (int k = 0; k < RP_CS; ++k) *cluster.map_shared_rank(&css[rank], k) = tot;
    }
    rp_cluster_arrive_release();
    rp_cluster_wait_acquire();   // every block's sum has arrived here
    float tot = 0.f;
#pragma unroll
    for (int k = 0; k < RP_CS; ++k) tot += css[k];
    const float inv = rsqrtf(tot / (float)a.nout + a.pl_eps);
    uint16_t *p0 = a.pl_dst + (size_t)prow * a.pl_ld + a.pl_col0;
    const size_t plane = (size_t)a.pl_npad * a.pl_ld;
#pragma unroll
    for (int i = 0; i < RP_VPT; ++i) {
        const int col = c0 + t + 256 * i;
        if (col >= c1) continue;
        const float v = act ? xv[i] * inv * bf_to_f(a.pl_gain[col]) : 0.f;
        uint16_t q[TC_PLANES];
        tc_split(v, q);
#pragma unroll
        for (int j = 0; j < TC_PLANES; ++j)
            if (j < a.pl_npl) p0[j * plane + col] = q[j];
    }
}

// ---------------------------------------------------------------- operand planes
// A block a row, and few rows: what bounds these kernels is the latency of a
// thread's chain of loads, so a row of d elements gets the width that leaves a
// thread four to eight of them.  With 256 threads at every d, a block drafter's
// call (d 4096, 120 rows) took 1902 us instead of 1884, a tree of 2048 wide
// rows 1905 instead of 1900; below d 2048 the width is what it was.
static int row_threads(int d) { return d >= 4096 ? 1024 : d >= 2048 ? 512 : 256; }
__global__ void __launch_bounds__(1024) planes_kernel(const PlaneArgs a) {
    __shared__ float red[33];
    const int r = blockIdx.x;
    pdl_trigger();
    pdl_wait();
    bool act;
    int srow;
    if (a.dec) {
        const int dr = __ldcg(&a.dec[a.dec_b0 + r].r);
        act = dr >= 0 && dr < a.dec_K;
        srow = act ? (a.dec_b0 + r) * a.dec_K + dr : 0;
    } else if (a.last_of_seq) {
        act = !a.valid || a.valid[r];
        srow = act ? r * a.max_new + a.nnew[r] - 1 : 0;
    } else {
        const int b = r / a.rows_per_seq, j = r - b * a.rows_per_seq;
        act = (!a.valid || a.valid[b]) && (a.rows_per_seq == 1 || j < a.nnew[b]);
        srow = r;
    }
    const float *x = a.src + (size_t)srow * a.d;
    float inv = 1.f;
    if (a.gain) {
        float ss = 0.f;
        if (act)
            for (int k = threadIdx.x; k < a.d; k += blockDim.x) ss = fmaf(x[k], x[k], ss);
        ss = warp_sum(ss);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
            red[32] = rsqrtf(t / (float)a.d + a.eps);
        }
        __syncthreads();
        inv = red[32];
    }
    uint16_t *p0 = a.dst + (size_t)r * a.ld + a.col0;
    const size_t plane = (size_t)a.npad * a.ld;
    const int npl = a.npl > 0 ? a.npl : TC_PLANES;
    for (int k = threadIdx.x; k < a.d; k += blockDim.x) {
        float v = act ? x[k] : 0.f;
        if (a.gain) v = v * inv * bf_to_f(a.gain[k]);
        uint16_t q[TC_PLANES];
        tc_split(v, q);
#pragma unroll
        for (int i = 0; i < TC_PLANES; ++i)
            if (i < npl) p0[i * plane + k] = q[i];
    }
    if (a.src2) {   // a second part of the row, copied without normalisation
        const float *x2 = a.src2 + (size_t)srow * a.d;
        uint16_t *p2 = a.dst + (size_t)r * a.ld + a.col2;
        for (int k = threadIdx.x; k < a.d; k += blockDim.x) {
            uint16_t q[TC_PLANES];
            tc_split(act ? x2[k] : 0.f, q);
#pragma unroll
            for (int i = 0; i < TC_PLANES; ++i)
                if (i < npl) p2[i * plane + k] = q[i];
        }
    }
}

// ---------------------------------------------------------------- RoPE + K/V write
__global__ void __launch_bounds__(256) qkv_post_kernel(const QkvPostArgs a) {
    const Dims &D = a.dim;
    const int half = D.hd / 2;
    const int per_row = (D.Hq + 2 * D.Hkv) * half;
    pdl_trigger();
    pdl_wait();
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)a.R * per_row) return;
    const int r = (int)(idx / per_row), item = (int)(idx % per_row);
    int b, pos;
    if (!a.map.row(r, b, pos)) return;
    const int h = item / half, ii = item % half;
    const float *yr = a.y + (size_t)r * (D.Hq + 2 * D.Hkv) * D.hd + (size_t)h * D.hd;
    float x1 = yr[ii], x2 = yr[ii + half];
    if (h < D.Hq + D.Hkv) {
        float c, sn;
        rope_cs2(a.inv_freq[ii], pos, c, sn);
        const float y1 = x1 * c - x2 * sn, y2 = x2 * c + x1 * sn;
        x1 = y1;
        x2 = y2;
    }
    if (h < D.Hq) {
        float *q = a.q + (size_t)r * D.Hq * D.hd + (size_t)h * D.hd;
        q[ii] = x1;
        q[ii + half] = x2;
    } else {
        const bool is_k = h < D.Hq + D.Hkv;
        const int kvh = is_k ? h - D.Hq : h - D.Hq - D.Hkv;
        const int page = a.page_table[(size_t)b * a.max_pages + pos / D.P];
        uint16_t *dst = (is_k ? a.k_pages : a.v_pages) + (((size_t)page * D.Hkv + kvh) * D.P + pos % D.P) * D.hd;
        dst[ii] = f_to_bf(x1);
        dst[ii + half] = f_to_bf(x2);
    }
}

// The QKV GEMM's split-K reduction with RoPE and the paged K/V write folded
// in: each thread sums the partials (in range order) of one rotary pair
// (ii, ii + hd / 2) of one head, then does what qkv_post_kernel does with it.
__global__ void __launch_bounds__(256) tc_reduce_rope_kernel(const TcArgs a, const QkvPostArgs p) {
    const Dims &D = p.dim;
    const int half = D.hd / 2;
    const int per_row = (D.Hq + 2 * D.Hkv) * half;
    pdl_trigger();
    pdl_wait();
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)a.R * per_row) return;
    const int r = (int)(idx / per_row), item = (int)(idx % per_row);
    int b, pos;
    if (!p.map.row(r, b, pos)) return;
    const int h = item / half, ii = item % half;
    const int col = h * D.hd + ii;
    float x1 = 0.f, x2 = 0.f;
    for (int sp = 0; sp < a.nsplit; ++sp) {
        const float *pr = a.part + ((size_t)sp * a.R + r) * a.nout;
        x1 += __ldcg(pr + col);
        x2 += __ldcg(pr + col + half);
    }
    if (h < D.Hq + D.Hkv) {
        float c, sn;
        rope_cs2(p.inv_freq[ii], pos, c, sn);
        const float y1 = x1 * c - x2 * sn, y2 = x2 * c + x1 * sn;
        x1 = y1;
        x2 = y2;
    }
    if (h < D.Hq) {
        float *q = p.q + (size_t)r * D.Hq * D.hd + (size_t)h * D.hd;
        q[ii] = x1;
        q[ii + half] = x2;
    } else {
        const bool is_k = h < D.Hq + D.Hkv;
        const int kvh = is_k ? h - D.Hq : h - D.Hq - D.Hkv;
        const int page = p.page_table[(size_t)b * p.max_pages + pos / D.P];
        uint16_t *dst = (is_k ? p.k_pages : p.v_pages) + (((size_t)page * D.Hkv + kvh) * D.P + pos % D.P) * D.hd;
        dst[ii] = f_to_bf(x1);
        dst[ii + half] = f_to_bf(x2);
    }
}

// ---------------------------------------------------------------- LM-head pick
constexpr int PK_THREADS = 1024, PK_WARPS = PK_THREADS / 32;
constexpr int PK_CH = 8;     // partials a lane holds (a row of 32 x 8 x 32 groups, V 262144; beyond, they are read again)
constexpr int PK_MAXK = 8;   // candidates per row at most

// Recomputes the 32 logits of each of n groups (ids 32 g ..): warp w takes id w of
// every group, two groups at a time, lanes split the reduction over the row's
// operand in shared memory.
__device__ __forceinline__ void pk_group_logits(const LmPickArgs &a, const float *hrow, const int *grp, int n, float *z) {
    const Dims &D = a.dim;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    static_assert(TC_LM_GROUP == PK_WARPS, "an id a warp");
    for (int q = 0; q < n; q += 2) {
        int id[2];
        const uint16_t *wr[2];
        float acc[2] = {0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            id[e] = q + e < n && grp[q + e] >= 0 ? grp[q + e] * TC_LM_GROUP + warp : D.V;
            wr[e] = a.W + (size_t)(id[e] < D.V ? id[e] : 0) * D.d + lane * 8;
        }
#pragma unroll 4
        for (int k = 0; k < D.d; k += 256) {   // (d is a multiple of 256)
            const uint4 w0 = ld_stream(wr[0] + k), w1 = q + 1 < n ? ld_stream(wr[1] + k) : make_uint4(0, 0, 0, 0);
            float f0[8], f1[8];
            unpack8(w0, f0);
            unpack8(w1, f1);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float h = hrow[k + lane * 8 + e];
                acc[0] = fmaf(f0[e], h, acc[0]);
                acc[1] = fmaf(f1[e], h, acc[1]);
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float v = warp_sum(acc[e]);
            if (lane == 0 && q + e < n) z[(q + e) * TC_LM_GROUP + warp] = id[e] < D.V ? v : -INFINITY;
        }
    }
}

// One block per row, bound by the latency of its steps: 64 rows of 6252 partials
// 12 us a launch, 16 rows with four greedy candidates 25 (17 and 37 when a thread
// walked a run of its own and every candidate cost passes over the partials).  Level 1: warp w holds the w-th contiguous range of the row's
// 32-id partials, lanes side by side (coalesced, all loads in flight), which gives
// M = max y, S = sum exp(y - M) and, per draw, the warp and then the group holding
// u * S.  Level 2: that group's 32 logits, recomputed as dot products of the
// LM-head rows with the row's operand (the sum of its bf16 planes), scanned in
// ascending ids.  Greedy: the argmax from the partials; with topk > 1 the next
// candidates come from the topk groups of largest maximum (the only groups
// that can hold one of the topk largest logits), recomputed together and ranked.
__global__ void __launch_bounds__(PK_THREADS) lm_pick_kernel(const LmPickArgs a) {
    extern __shared__ float hrow[];   // [d] the row's LM-head operand
    __shared__ AM sm_am[2][PK_WARPS];
    __shared__ float sm_m[PK_WARPS], sm_w[PK_WARPS], sh[PK_WARPS];
    __shared__ float s_z[PK_MAXK * TC_LM_GROUP];
    __shared__ int s_grp[PK_MAXK], s_tok[PK_MAXK];
    __shared__ float s_before, s_e[PK_MAXK];
    const Dims &D = a.dim;
    const int b = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int topk = a.topk > 1 ? a.topk : 1;
    pdl_trigger();
    pdl_wait();
    if (!a.valid[b]) return;
    const bool greedy = a.temperature == 0.f;
    const float invT = greedy ? 1.f : 1.f / a.temperature;
    const float4 *pp = a.part + (size_t)b * a.nsub;
    const int per = ((a.nsub + PK_WARPS - 1) / PK_WARPS + 31) / 32 * 32;   // partials of a warp
    const int j0 = min(a.nsub, warp * per), j1 = min(a.nsub, j0 + per);
    const int nch = (j1 - j0 + 31) / 32;                                   // of a lane
    float px[PK_CH], py[PK_CH];
    float m = -INFINITY;
    AM am{-INFINITY, 0x7fffffff};
    {
        float4 v[PK_CH];
#pragma unroll
        for (int i = 0; i < PK_CH; ++i) {
            const int j = j0 + 32 * i + lane;
            v[i] = j < j1 ? __ldcg(pp + j) : make_float4(-INFINITY, 0.f, -INFINITY, __int_as_float(0x7fffffff));
        }
        // meanwhile: the row's operand, the sum of its planes (the values the tensor
        // cores multiplied), and the next chain row's context slot, x_L (Sec. 3.4)
        if (topk > 1 || !greedy) {
            const size_t plane = (size_t)a.npad * D.d;
            const uint16_t *q = a.planes + (size_t)b * D.d;
            for (int k = t; k < D.d; k += PK_THREADS) {
                float h = 0.f;
#pragma unroll
                for (int i = 0; i < TC_PLANES; ++i)
                    if (i < a.npl) h += bf_to_f(q[i * plane + k]);
                hrow[k] = h;
            }
        }
        if (a.step + 1 < a.K) {
            const int src = a.src_is_ext ? b * a.max_new + a.nnew[b] - 1 : b;
            const float *xl = a.x_in + (size_t)src * D.d;
            const size_t ld = 2 * (size_t)D.d, plane = (size_t)a.qkv_npad * ld;
            for (int k = t; k < D.d; k += PK_THREADS) {
                const float x = xl[k];
                a.s_chain[(size_t)b * D.d + k] = x;
                if (a.qkv_planes) {
                    uint16_t q[TC_PLANES];
                    tc_split(x, q);
#pragma unroll
                    for (int i = 0; i < TC_PLANES; ++i) a.qkv_planes[(size_t)b * ld + i * plane + k] = q[i];
                }
            }
        }
#pragma unroll
        for (int i = 0; i < PK_CH; ++i) {
            px[i] = v[i].x;
            py[i] = v[i].y;
            m = fmaxf(m, v[i].x);
            am = am_combine(am, AM{v[i].z, __float_as_int(v[i].w)});
        }
    }
    for (int i = PK_CH; i < nch; ++i) {
        const int j = j0 + 32 * i + lane;
        if (j >= j1) break;
        const float4 p = __ldcg(pp + j);
        m = fmaxf(m, p.x);
        am = am_combine(am, AM{p.z, __float_as_int(p.w)});
    }
    m = warp_max(m);
    if (greedy) am = warp_am(am);
    if (lane == 0) {
        sm_m[warp] = m;
        sm_am[0][warp] = am;
    }
    __syncthreads();
    const float M = warp_max(sm_m[lane]);
    auto weight = [&](float x, float y) { return x == -INFINITY ? 0.f : y * __expf(x - M); };
    // partial i of the lane: its weight (and for i >= PK_CH its place again from memory)
    float mine = 0.f;
#pragma unroll
    for (int i = 0; i < PK_CH; ++i) {
        py[i] = weight(px[i], py[i]);
        mine += py[i];
    }
    auto far = [&](int i) {
        const int j = j0 + 32 * i + lane;
        const float4 p = j < j1 ? __ldcg(pp + j) : make_float4(-INFINITY, 0.f, 0.f, 0.f);
        return make_float2(p.x, weight(p.x, p.y));
    };
    for (int i = PK_CH; i < nch; ++i) mine += far(i).y;
    mine = warp_sum(mine);
    if (lane == 0) sm_w[warp] = mine;
    __syncthreads();
    const float wtot = sm_w[lane], wincl = warp_incl_scan(wtot);   // lane k: warp k's range
    const float S = __shfl_sync(0xffffffffu, wincl, 31);
    if (greedy) {
        const AM top = warp_am(sm_am[0][lane]);   // candidate 0: the argmax of the tensor-core logits
        if (t == 0) { s_tok[0] = top.i; s_e[0] = 1.f; }
        if (topk > 1) {
            // the topk groups of largest maximum, one block argmax per round
            int taken[PK_MAXK];
#pragma unroll
            for (int r = 0; r < PK_MAXK; ++r) {
                if (r >= topk) break;
                AM loc{-INFINITY, 0x7fffffff};
                auto offer = [&](float x, int j) {
                    bool was = j >= j1;
#pragma unroll
                    for (int rr = 0; rr < r; ++rr) was |= taken[rr] == j;
                    if (!was) loc = am_combine(loc, AM{x, j});
                };
#pragma unroll
                for (int i = 0; i < PK_CH; ++i) offer(px[i], j0 + 32 * i + lane);
                for (int i = PK_CH; i < nch; ++i) offer(far(i).x, j0 + 32 * i + lane);
                loc = warp_am(loc);
                AM *slot = sm_am[(r + 1) & 1];   // in turn: one barrier a round
                if (lane == 0) slot[warp] = loc;
                __syncthreads();
                const AM g = warp_am(slot[lane]);
                taken[r] = g.v == -INFINITY ? -1 : g.i;
                if (t == 0) s_grp[r] = taken[r];
            }
            __syncthreads();
            pk_group_logits(a, hrow, s_grp, topk, s_z);
            __syncthreads();
            // rank: candidates 1.. are the largest recomputed logits other than candidate 0
            if (warp == 0) {
                float z[PK_MAXK];
#pragma unroll
                for (int r = 0; r < PK_MAXK; ++r) z[r] = r < topk ? s_z[r * TC_LM_GROUP + lane] : -INFINITY;
                int last = top.i;
                for (int c = 1; c < topk; ++c) {
                    AM loc{-INFINITY, 0x7fffffff};
#pragma unroll
                    for (int r = 0; r < PK_MAXK; ++r) {
                        const int id = r < topk && s_grp[r] >= 0 ? s_grp[r] * TC_LM_GROUP + lane : -1;
                        if (id < 0 || id == last) z[r] = -INFINITY;   // taken
                        else loc = am_combine(loc, AM{z[r], id});
                    }
                    const AM best = warp_am(loc);
                    // no finite logit left: candidate 0 again
                    last = best.v == -INFINITY ? -1 : best.i;
                    if (lane == 0) { s_tok[c] = best.v == -INFINITY ? top.i : best.i; s_e[c] = 1.f; }
                }
            }
        }
        __syncthreads();
    } else {
        // each draw: its warp and group from the partials, then its id inside the recomputed group
        for (int c = 0; c < topk; ++c) {
            const float target = a.u_draft[((size_t)b * a.K + a.step) * topk + c] * S;
            const unsigned hits = __ballot_sync(0xffffffffu, wtot > 0.f && target < wincl);
            const unsigned some = __ballot_sync(0xffffffffu, wtot > 0.f);
            const int ct = hits ? __ffs(hits) - 1 : (some ? 31 - __clz(some) : 0);
            const float before = __shfl_sync(0xffffffffu, wincl - wtot, ct);
            if (warp == ct) {   // this warp's range holds the point: find its group
                float run = before, bef = before;
                int grp = -1, lastg = j0;
                float lastb = before;
                auto walk = [&](int i, float w) {   // warp-uniform but for w
                    const float incl = warp_incl_scan(w);
                    const unsigned h = __ballot_sync(0xffffffffu, w > 0.f && target < run + incl);
                    const unsigned pos = __ballot_sync(0xffffffffu, w > 0.f);
                    if (h) {
                        const int l = __ffs(h) - 1;
                        grp = j0 + 32 * i + l;
                        bef = run + __shfl_sync(0xffffffffu, incl - w, l);
                    } else if (pos) {
                        const int l = 31 - __clz(pos);
                        lastg = j0 + 32 * i + l;
                        lastb = run + __shfl_sync(0xffffffffu, incl - w, l);
                    }
                    run += __shfl_sync(0xffffffffu, incl, 31);
                };
#pragma unroll
                for (int i = 0; i < PK_CH; ++i)
                    if (grp < 0) walk(i, py[i]);
                for (int i = PK_CH; i < nch && grp < 0; ++i) walk(i, far(i).y);
                if (lane == 0) {
                    s_grp[c] = grp >= 0 ? grp : lastg;
                    s_before = grp >= 0 ? bef : lastb;
                }
            }
            __syncthreads();
            // Batches whose logits were float32 sums before (three planes): M is off by a few
            // 1e-6 against the recomputed logits, and so would q be (1 + 7e-6 for a token of
            // all the mass).  The group is scaled to its partial, which M and S come from.
            const bool scaled = a.npl > TC_LM_PLANES;
            const float4 part = scaled ? __ldcg(pp + s_grp[c]) : make_float4(0.f, 0.f, 0.f, 0.f);
            pk_group_logits(a, hrow, s_grp + c, 1, s_z);
            __syncthreads();
            if (warp == 0) {
                const int id = s_grp[c] * TC_LM_GROUP + lane;
                float e = id < D.V ? __expf(s_z[lane] * invT - M) : 0.f;
                if (scaled) {
                    const float mass = weight(part.x, part.y), sum = warp_sum(e);
                    if (mass > 0.f && sum > 0.f) e *= mass / sum;
                }
                const float cum = s_before + warp_incl_scan(e);
                const unsigned hit = __ballot_sync(0xffffffffu, e > 0.f && target < cum);
                const unsigned pos = __ballot_sync(0xffffffffu, e > 0.f);
                const int l = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
                if (lane == l) { s_tok[c] = id; s_e[c] = e; }
            }
            __syncthreads();
        }
    }
    const size_t o = (size_t)b * a.K + a.step;
    if (t < topk) {
        a.tokens[o * topk + t] = s_tok[t];
        if (a.qx) a.qx[o * topk + t] = greedy ? 1.f : s_e[t] / S;
    }
    if (t == 0 && a.stats) {
        a.stats[o * 2 + 0] = M;
        a.stats[o * 2 + 1] = logf(S);
    }
    const int token = min(max(s_tok[0], 0), D.V - 1);   // a row of NaN has no argmax
    if (a.step + 1 < a.K) {
        // next chain row: residual <- E[candidate 0] (its context slot was written above;
        // x_in may be x_chain, and every thread overwrites only what it has read)
        const uint16_t *er = a.embed + (size_t)token * D.d;
        float ss = 0.f;
        for (int k = t; k < D.d; k += PK_THREADS) {
            const float e = bf_to_f(er[k]);
            a.x_chain[(size_t)b * D.d + k] = e;
            ss = fmaf(e, e, ss);
        }
        if (a.qkv_planes) {   // and its first layer's operand's second half, RMSNorm(x)
            ss = warp_sum(ss);
            if (lane == 0) sh[warp] = ss;
            __syncthreads();
            const float inv = rsqrtf(warp_sum(sh[lane]) / (float)D.d + a.eps);
            const size_t ld = 2 * (size_t)D.d, plane = (size_t)a.qkv_npad * ld;
            uint16_t *p0 = a.qkv_planes + (size_t)b * ld;
            for (int k = t; k < D.d; k += PK_THREADS) {
                uint16_t q[TC_PLANES];
                tc_split(bf_to_f(er[k]) * inv * bf_to_f(a.qkv_gain[k]), q);
#pragma unroll
                for (int i = 0; i < TC_PLANES; ++i) p0[i * plane + D.d + k] = q[i];
            }
        }
    }
}

// The draw of a block row (row b of sequence b / max_new, one candidate, no next
// step): the partials as contiguous runs, one a thread, summed and scanned in the
// order that block drafting keeps (see TcArgs::block).  120 rows of 4748 partials,
// d 4096: 19 us a launch.
__global__ void __launch_bounds__(PK_THREADS) block_pick_kernel(const LmPickArgs a) {
    extern __shared__ float hrow[];   // [d] the row's LM-head operand
    __shared__ MS sm_ms[PK_WARPS];
    __shared__ AM sm_am[PK_WARPS];
    __shared__ float sh[34], s_z[TC_LM_GROUP], s_before;
    __shared__ int si[2], s_grp;
    const Dims &D = a.dim;
    const int b = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    pdl_trigger();
    pdl_wait();
    if (!a.valid[b / a.max_new]) return;
    const bool greedy = a.temperature == 0.f;
    const float invT = greedy ? 1.f : 1.f / a.temperature;
    const float4 *pp = a.part + (size_t)b * a.nsub;
    const int per = (a.nsub + PK_THREADS - 1) / PK_THREADS;
    const int j0 = min(a.nsub, t * per), j1 = min(a.nsub, j0 + per);
    // the run's argmax, and its (max, sum) rescaled online
    float m = -INFINITY, sm = 0.f;
    AM am{-INFINITY, 0x7fffffff};
    for (int j = j0; j < j1; ++j) {
        const float4 p = __ldcg(pp + j);
        am = am_combine(am, AM{p.z, __float_as_int(p.w)});
        if (p.x == -INFINITY) continue;
        if (p.x > m) {
            sm = (m == -INFINITY ? 0.f : sm * __expf(m - p.x)) + p.y;
            m = p.x;
        } else {
            sm += p.y * __expf(p.x - m);
        }
    }
    const MS tot = block_ms(MS{m, sm}, sm_ms);
    const float M = tot.m, S = tot.s;
    if (greedy) {
        const AM top = block_am(am, sm_am);
        if (t == 0) {
            a.tokens[b] = top.i;
            if (a.qx) a.qx[b] = 1.f;
        }
    } else {
        const float w = m == -INFINITY ? 0.f : sm * __expf(m - M);   // the run's weight
        const size_t plane = (size_t)a.npad * D.d;
        const uint16_t *q = a.planes + (size_t)b * D.d;
        for (int k = t; k < D.d; k += PK_THREADS) {
            float h = 0.f;
#pragma unroll
            for (int i = 0; i < TC_LM_PLANES; ++i) h += bf_to_f(q[i * plane + k]);
            hrow[k] = h;
        }
        float all;
        const float ex = block_excl_scan(w, sh, &all);
        const float target = a.u_draft[b] * S;
        if (t == 0) { si[0] = 0x7fffffff; si[1] = -1; }
        __syncthreads();
        if (w > 0.f && target < ex + w) atomicMin(&si[0], t);
        if (w > 0.f) atomicMax(&si[1], t);
        __syncthreads();
        const int ct = si[0] != 0x7fffffff ? si[0] : (si[1] >= 0 ? si[1] : 0);
        if (t == ct) {   // this thread's run holds the point: find its group
            float cum = ex;
            int grp = -1, lastg = -1;
            float lastb = ex;
            for (int j = j0; j < j1; ++j) {
                const float4 p = __ldcg(pp + j);
                const float wj = p.x != -INFINITY ? p.y * __expf(p.x - M) : 0.f;
                if (wj > 0.f) { lastg = j; lastb = cum; }
                if (wj > 0.f && target < cum + wj) { grp = j; break; }
                cum += wj;
            }
            s_grp = grp >= 0 ? grp : (lastg >= 0 ? lastg : j0);
            s_before = grp >= 0 ? cum : lastb;
        }
        __syncthreads();
        pk_group_logits(a, hrow, &s_grp, 1, s_z);
        __syncthreads();
        if (warp == 0) {
            const int id = s_grp * TC_LM_GROUP + lane;
            const float e = id < D.V ? __expf(s_z[lane] * invT - M) : 0.f;
            const float cum = s_before + warp_incl_scan(e);
            const unsigned hit = __ballot_sync(0xffffffffu, e > 0.f && target < cum);
            const unsigned pos = __ballot_sync(0xffffffffu, e > 0.f);
            const int l = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
            if (lane == l) {
                a.tokens[b] = id;
                if (a.qx) a.qx[b] = e / S;
            }
        }
    }
    if (t == 0 && a.stats) {
        a.stats[(size_t)b * 2 + 0] = M;
        a.stats[(size_t)b * 2 + 1] = logf(S);
    }
}

// ---------------------------------------------------------------- embedding rows
__global__ void __launch_bounds__(1024) embed_rows_kernel(const EmbedArgs a) {
    const int r = blockIdx.x, b = r / a.max_new, j = r - b * a.max_new;
    pdl_trigger();
    pdl_wait();
    if (!a.valid[b] || j >= a.nnew[b]) return;
    const uint16_t *e = a.embed + (size_t)a.tokens[r] * a.d;   // ids checked by the prepare kernel
    for (int k = threadIdx.x; k < a.d; k += blockDim.x) a.x[(size_t)r * a.d + k] = bf_to_f(e[k]);
}

// ---------------------------------------------------------------- block inputs
__global__ void __launch_bounds__(256) block_inputs_kernel(const BlockInArgs a) {
    const int r = blockIdx.x, b = r / a.P, j = r - b * a.P;
    if (threadIdx.x == 0) {
        a.tokens[r] = j == 0 ? a.anchors[b] : a.mask;
        if (j == 0) a.nnew[b] = a.P;
    }
    const uint4 *src = (const uint4 *)(a.feats + (size_t)b * a.feat);
    uint4 *dst = (uint4 *)(a.feats_rep + (size_t)r * a.feat);
    for (int k = threadIdx.x; k < a.feat / 8; k += blockDim.x) dst[k] = src[k];
}

cudaError_t launch_block_inputs(const BlockInArgs &a, cudaStream_t s) {
    // a normal launch: the draft call's prepare kernel reads these arrays
    block_inputs_kernel<<<a.n * a.P, 256, 0, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------- host side
static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

// The driver's tensor-map encoder and a device with tcgen05 (compute
// capability 10 or above); looked up once, thread-safely (a function-local
// static is initialised exactly once).
bool tc_available() {
    static const bool ok = [] {
        cudaDriverEntryPointQueryResult q;
        void *fn = nullptr;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        g_encode = e == cudaSuccess && q == cudaDriverEntryPointSuccess ? (PFN_cuTensorMapEncodeTiled_v12000)fn : nullptr;
        if (e != cudaSuccess) cudaGetLastError();
        int dev = 0, major = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) {
            cudaGetLastError();
            major = 0;
        }
        return g_encode != nullptr && major >= 10;
    }();
    return ok;
}

static bool encode2d(CUtensorMap *m, const void *base, uint64_t inner, uint64_t rows, uint32_t box_rows) {
    if (!tc_available()) return false;
    if (((uintptr_t)base & 15) || (inner * 2) % 16) return false;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)inner * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t es[2] = {1, 1};
    return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tc_encode_weight(CUtensorMap *m, const void *w, int rows, int K) { return encode2d(m, w, K, rows, 128); }
bool tc_encode_rows(CUtensorMap *m, const void *x, int rows, int npad, int K) { return encode2d(m, x, K, rows, npad); }
bool tc_encode_operand(CUtensorMap *m, const void *x, int planes, int prows, int npad, int K) {
    return encode2d(m, x, K, (uint64_t)planes * prows, npad);
}

static int tc_stages(int npad, int planes, int na, int bps) {
    const size_t stage = (size_t)na * TC_ABYTES + (size_t)planes * npad * 128;
    int n = (int)((tc_smem_cap(bps) - 1024) / stage);
    return n > TC_MAXST ? TC_MAXST : n;
}
static size_t tc_smem_bytes(int npad, int planes, int na, int bps) {
    const size_t stage = (size_t)na * TC_ABYTES + (size_t)planes * npad * 128;
    return (size_t)tc_stages(npad, planes, na, bps) * stage + 1024;
}

cudaError_t tc_set_attributes() {
    const cudaError_t e = allow_smem(lm_pick_kernel);
    return e == cudaSuccess ? allow_smem(block_pick_kernel) : e;
}

template <typename... P, typename... A>
static cudaError_t pdl_launch(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, args...);
    count_launch();
    return e;
}

template <int EPI, int NA, int BPS>
static cudaError_t tc_launch(int grid, size_t smem, cudaStream_t s, const CUtensorMap &wa, const CUtensorMap &wb,
                             const CUtensorMap &xm, const TcArgs &a, int nst) {
    // opted into its shared memory, and so loaded, at its first launch: with every
    // instance loaded beside them, calls that use none (one sequence, batch-1 weights
    // in L2) took 678 us instead of 673
    static std::atomic<int> done[kMaxDevices];
    const cudaError_t es = once_per_device(done, [] {
        return cudaFuncSetAttribute(tc_kernel<EPI, NA, BPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)tc_smem_cap(BPS));
    });
    if (es != cudaSuccess) return es;
    return pdl_launch(tc_kernel<EPI, NA, BPS>, dim3(grid), dim3(TC_THREADS), smem, s, wa, wb, xm, a, nst);
}

cudaError_t launch_tc(const TcArgs &a_in, const CUtensorMap &wa, const CUtensorMap &xm, int sms, cudaStream_t s) {
    TcArgs a = a_in;
    a.nout_a = a.nout;
    return launch_tc2(a, wa, wa, xm, sms, s);
}

cudaError_t launch_tc2(const TcArgs &a_in, const CUtensorMap &wa, const CUtensorMap &wb, const CUtensorMap &xm, int sms,
                       cudaStream_t s, bool *planes_done, const QkvPostArgs *rope) {
    TcArgs a = a_in;
    if (planes_done) *planes_done = false;
    if (a.nrt < 1) a.nrt = 1;
    if (a.bps != 1) a.bps = 2;
    const bool lm = a.epi == TC_LM || a.epi == TC_LM_BLOCK;
    if (a.prows < 1) a.prows = a.nrt * a.npad;
    if (a.bps == 1 && lm) return cudaErrorInvalidValue;
    if (a.npad % 16 || a.npad < 16 || a.npad > (a.bps == 1 ? TC_BIG_ROWS : TC_TILE_ROWS) || a.K % 64 || a.R > (long long)a.nrt * a.npad)
        return cudaErrorInvalidValue;
    if (a.nout_a < 1 || a.nout_a > a.nout || (a.nout_a < a.nout && a.nout_a % 128)) return cudaErrorInvalidValue;
    if (a.epi == TC_GLU && (a.nout != 2 * a.nout_a || !a.part || !a.h || a.h_rows < a.R)) return cudaErrorInvalidValue;
    const int nkb = a.K / 64;
    if (lm && (!a.lm_part || a.lm_nsub != (a.nout + TC_LM_GROUP - 1) / TC_LM_GROUP))
        return cudaErrorInvalidValue;
    // (the LM epilogue needs whole sums)
    a.nsplit = a.part && !lm ? tc_nsplit(a.nout, a.K, a.block ? TC_BLOCK_SPLITS : TcTiles{a.nrt, a.npad, a.bps}, sms) : 1;
    if ((long long)a.nsplit * a.R * a.nout > a.part_cap) a.nsplit = 1;
    if (a.epi == TC_GLU && (long long)a.nsplit * a.R * a.nout > a.part_cap) return cudaErrorInvalidValue;
    a.kbps = (nkb + a.nsplit - 1) / a.nsplit;
    a.sep = a.planes > 1 && !a.block;   // (0.1 % of a call, for a third of the accumulators' error)
    a.segkb = !a.fine ? OSP_TC_SEGKB : lm ? OSP_TC_SEGKB_LM : OSP_TC_SEGKB_FINE;
    const int bps = a.bps, tmem_cols = tc_tmem_cols(bps);
    // the LM head takes OSP_TC_LM_NA weight tiles per stage when two stages fit
    // and the double-buffered accumulators fit TMEM in one segment (the LM head's
    // reduction over d is short: one segment keeps its MMA chain at 4 d / 64 steps
    // per plane)
    int na = 1;
    if (a.block && a.whole) a.segkb = a.kbps;
    const bool wide = (lm && (!a.block || a.whole)) || (a.epi == TC_STORE && a.nsplit == 1 && a.wide);
    if (wide && a.nrt == 1 && OSP_TC_LM_NA > 1 && tc_stages(a.npad, a.planes, OSP_TC_LM_NA, bps) >= 2 &&
        2 * OSP_TC_LM_NA * a.npad <= tmem_cols && a.kbps <= 32 && a.planes <= TC_LM_PLANES) {
        na = OSP_TC_LM_NA;
        a.segkb = a.kbps;
    }
    const int nst = tc_stages(a.npad, a.planes, na, bps);
    if (nst < 2) return cudaErrorInvalidValue;
    if ((na == 1 && a.sep ? 3 : 2) * na * a.npad > tmem_cols) return cudaErrorInvalidValue;   // TMEM columns
    // an even number of row tiles goes in pairs: the weights of the second one come from
    // L2 also where a tile's next one would find them gone (120 rows, d 4096: 2496 us a
    // call, one row tile after the other 2570; 96 rows, d 1024: 2864, 2884)
    a.pair = a.nrt % 2 == 0 ? 2 : 1;
    const int items = (a.nout + 128 * na - 1) / (128 * na) * (a.nrt / a.pair) * a.nsplit, slots = bps * sms / a.pair;
    const int grid = (items < slots ? items : slots) * a.pair;
    const size_t smem = tc_smem_bytes(a.npad, a.planes, na, bps);
    cudaError_t e;
#define OSP_TC_GO(EPI, NA_, BPS_) tc_launch<EPI, NA_, BPS_>(grid, smem, s, wa, wb, xm, a, nst)
#define OSP_TC_ROWS(EPI) (bps == 1 ? OSP_TC_GO(EPI, 1, 1) : OSP_TC_GO(EPI, 1, 2))
    switch (a.epi) {
    case TC_STORE: e = na > 1 ? OSP_TC_GO(TC_STORE, OSP_TC_LM_NA, 2) : OSP_TC_ROWS(TC_STORE); break;
    case TC_RESID: e = OSP_TC_ROWS(TC_RESID); break;
    case TC_GLU: e = OSP_TC_ROWS(TC_GLU); break;
    case TC_LM_BLOCK: e = na > 1 ? OSP_TC_GO(TC_LM_BLOCK, OSP_TC_LM_NA, 2) : OSP_TC_GO(TC_LM_BLOCK, 1, 2); break;
    default: e = na > 1 ? OSP_TC_GO(TC_LM, OSP_TC_LM_NA, 2) : OSP_TC_GO(TC_LM, 1, 2); break;
    }
#undef OSP_TC_ROWS
#undef OSP_TC_GO
    if (e != cudaSuccess || (a.nsplit == 1 && a.epi != TC_GLU)) return e;
    if (a.epi == TC_RESID && a.pl_dst && a.nout <= RP_CS * 256 * RP_VPT) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(RP_CS, a.R);
        cfg.blockDim = dim3(256);
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = RP_CS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        e = cudaLaunchKernelEx(&cfg, tc_resid_planes_kernel, a);
        count_launch();
        if (e == cudaSuccess && planes_done) *planes_done = true;
        return e;
    }
    if (a.epi == TC_STORE && rope) {
        const long long n = (long long)a.R * (rope->dim.Hq + 2 * rope->dim.Hkv) * (rope->dim.hd / 2);
        e = pdl_launch(tc_reduce_rope_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, a, *rope);
        if (e == cudaSuccess && planes_done) *planes_done = true;
        return e;
    }
    const unsigned rblocks =
        (unsigned)(((long long)a.R * (a.epi == TC_GLU ? a.nout_a : a.nout) + 255) / 256);
    switch (a.epi) {
    case TC_STORE: return pdl_launch(tc_reduce_kernel<TC_STORE>, dim3(rblocks), dim3(256), 0, s, a);
    case TC_RESID: return pdl_launch(tc_reduce_kernel<TC_RESID>, dim3(rblocks), dim3(256), 0, s, a);
    default: return pdl_launch(tc_reduce_kernel<TC_GLU>, dim3(rblocks), dim3(256), 0, s, a);
    }
}

cudaError_t launch_planes(const PlaneArgs &a, cudaStream_t s) {
    return pdl_launch(planes_kernel, dim3(a.R), dim3(a.block ? 256 : row_threads(a.d)), 0, s, a);
}

cudaError_t launch_qkv_post(const QkvPostArgs &a, cudaStream_t s) {
    const long long n = (long long)a.R * (a.dim.Hq + 2 * a.dim.Hkv) * (a.dim.hd / 2);
    return pdl_launch(qkv_post_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, a);
}

cudaError_t launch_embed_rows(const EmbedArgs &a, cudaStream_t s) {
    return pdl_launch(embed_rows_kernel, dim3(a.R), dim3(row_threads(a.d)), 0, s, a);
}

cudaError_t launch_lm_pick(const LmPickArgs &a, cudaStream_t s) {
    return pdl_launch(lm_pick_kernel, dim3(a.B), dim3(PK_THREADS), (size_t)a.dim.d * 4, s, a);
}

cudaError_t launch_block_pick(const LmPickArgs &a, cudaStream_t s) {
    return pdl_launch(block_pick_kernel, dim3(a.B), dim3(PK_THREADS), (size_t)a.dim.d * 4, s, a);
}

}  // namespace osp
