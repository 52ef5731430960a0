// Paged KV-cache append: scatter caller-provided K/V rows into the pages after
// each sequence's committed length, then advance the committed lengths.
#include "common.cuh"
#include "internal.h"
#include "tma.cuh"

namespace osp {

constexpr int KV_THREADS = 256;
constexpr int KV_GROUP = 16;       // rows a block copies together
constexpr int KV_FLIGHT = 8;       // 16-byte loads of a thread in flight
constexpr int KV_BLOCKS_PER_SM = 4;

// Exclusive prefix of one int64 per thread over the block; *total: the sum.
__device__ __forceinline__ int64_t kv_block_scan(int64_t v, int64_t *sh, int64_t *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) sh[w] = inc;
    __syncthreads();
    int64_t before = 0, tot = 0;
#pragma unroll
    for (int k = 0; k < KV_THREADS / 32; ++k) {
        if (k < w) before += sh[k];
        tot += sh[k];
    }
    __syncthreads();
    *total = tot;
    return before + inc - v;
}

// Bound by memory: every row is read once and written once.  Persistent blocks,
// each with a contiguous range of the flattened rows: a block rebuilds the
// per-sequence row offsets once, by a scan over the batch, then copies KV_GROUP
// rows at a time, their owners and pages looked up by one thread a row,
// KV_FLIGHT loads of a thread in flight.  67 k rows of 32 sequences, 4 KB a row
// (553 MB moved): 100 us with kv_advance, 5.6 TB/s; when one thread of every
// 8-row block walked the counts and one thread a sequence checked its pages, 212.
__global__ void __launch_bounds__(KV_THREADS, KV_BLOCKS_PER_SM) kv_scatter(KvAppendArgs a) {
    extern __shared__ int64_t off[];            // [B + 1] first row of each sequence
    __shared__ int64_t sh[KV_THREADS / 32];
    __shared__ int64_t s_dst[KV_GROUP];         // element offset of the row's first head inside a layer's pages, -1: skip
    const int64_t r0 = a.total_rows * blockIdx.x / gridDim.x, r1 = a.total_rows * (blockIdx.x + 1) / gridDim.x;
    const int per = (a.B + KV_THREADS - 1) / KV_THREADS;
    const int b0 = min(a.B, (int)threadIdx.x * per), b1 = min(a.B, b0 + per);
    int64_t mine = 0, total;
    int neg = 0;
    for (int b = b0; b < b1; ++b) {
        const int n = a.n_rows[b];
        neg |= n < 0;
        mine += n;
    }
    int64_t at = kv_block_scan(mine, sh, &total);
    for (int b = b0; b < b1; ++b) {
        off[b] = at;
        at += a.n_rows[b];
    }
    if (threadIdx.x == 0) off[a.B] = total;
    if (__syncthreads_or(neg) || total != a.total_rows) return;   // reported by kv_advance
    pdl_trigger();
    const int rowc = a.Hkv * a.hd / 8;          // 16-byte pieces of one row of one layer
    const int headc = a.hd / 8;                 // ... of one head
    const size_t layer_rows = (size_t)a.total_rows * a.Hkv * a.hd;
    const size_t layer_pages = (size_t)a.n_pages * a.Hkv * a.P * a.hd;
    for (int64_t g = r0; g < r1; g += KV_GROUP) {
        const int rows = (int)min((int64_t)KV_GROUP, r1 - g);
        if ((int)threadIdx.x < rows) {
            const int64_t r = g + threadIdx.x;
            int lo = 0, hi = a.B - 1;           // owner: last b with off[b] <= r
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (off[mid] <= r) lo = mid; else hi = mid - 1;
            }
            const int64_t n = off[lo + 1] - off[lo];
            const int L0 = a.seq_len[lo];
            const int64_t pos = (int64_t)L0 + (r - off[lo]);
            int64_t d = -1;
            if (L0 >= 0 && (int64_t)L0 + n <= (int64_t)a.max_pages * a.P) {
                const int page = a.page_table[(size_t)lo * a.max_pages + pos / a.P];
                if (page >= 0 && page < a.n_pages) d = ((int64_t)page * a.Hkv * a.P + pos % a.P) * a.hd;
            }
            s_dst[threadIdx.x] = d;
        }
        __syncthreads();
        const int pieces = rows * rowc;         // of one layer's K (or V) of the group: contiguous in the source
        for (int lk = 0; lk < 2 * a.L; ++lk) {
            const int l = lk >> 1;
            const uint16_t *src = (const uint16_t *)(lk & 1 ? a.v_rows : a.k_rows) + l * layer_rows + (size_t)g * rowc * 8;
            uint16_t *dst = (uint16_t *)(lk & 1 ? a.v_pages : a.k_pages) + l * layer_pages;
            for (int c0 = threadIdx.x; c0 < pieces; c0 += KV_THREADS * KV_FLIGHT) {
                uint4 v[KV_FLIGHT];
#pragma unroll
                for (int i = 0; i < KV_FLIGHT; ++i) {
                    const int c = c0 + i * KV_THREADS;
                    if (c < pieces) v[i] = ld_stream(src + (size_t)c * 8);
                }
#pragma unroll
                for (int i = 0; i < KV_FLIGHT; ++i) {
                    const int c = c0 + i * KV_THREADS;
                    if (c >= pieces) break;
                    const int row = c / rowc, hc = c - row * rowc, h = hc / headc;
                    const int64_t d = s_dst[row];
                    if (d >= 0) *(uint4 *)(dst + d + (size_t)h * a.P * a.hd + (hc - h * headc) * 8) = v[i];
                }
            }
        }
        __syncthreads();
    }
}

// Checks the row counts, then advances each sequence whose rows all fit
// (capacity and valid page ids); reports a failure in *status.  One warp a
// sequence, its lanes over the sequence's pages; the checks run while the
// scatter copies (it changes nothing that they read).
__global__ void __launch_bounds__(KV_THREADS) kv_advance(KvAppendArgs a) {
    __shared__ int64_t sh[KV_THREADS / 32];
    int64_t mine = 0, total;
    int neg = 0;
    for (int b = threadIdx.x; b < a.B; b += KV_THREADS) {
        const int n = a.n_rows[b];
        neg |= n < 0;
        mine += n;
    }
    kv_block_scan(mine, sh, &total);
    if (__syncthreads_or(neg) || total != a.total_rows) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_status(a.status, OSPREY_ERR_INVALID_ARG);
        return;
    }
    const int b = blockIdx.x * (KV_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const bool act = b < a.B;
    int n = 0, L0 = 0;
    bool ok = true;
    if (act) {
        n = a.n_rows[b];
        L0 = a.seq_len[b];
        ok = L0 >= 0 && (int64_t)L0 + n <= (int64_t)a.max_pages * a.P;
        if (ok && n > 0) {
            const int last = (L0 + n - 1) / a.P;
            for (int pg = L0 / a.P + lane; pg <= last; pg += 32) {
                const int page = a.page_table[(size_t)b * a.max_pages + pg];
                ok &= page >= 0 && page < a.n_pages;
            }
        }
    }
    ok = __all_sync(0xffffffffu, ok);
    pdl_wait();   // the scatter has read every sequence's committed length
    if (!act || lane) return;
    if (ok) a.seq_len[b] = L0 + n;
    else set_status(a.status, OSPREY_ERR_CAPACITY);
}

cudaError_t launch_kv_append(const KvAppendArgs &a, cudaStream_t s) {
    if (a.total_rows > 0) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const int64_t groups = (a.total_rows + KV_GROUP - 1) / KV_GROUP, cap = (int64_t)KV_BLOCKS_PER_SM * sms;
        kv_scatter<<<(unsigned)(groups < cap ? groups : cap), KV_THREADS, (size_t)(a.B + 1) * sizeof(int64_t), s>>>(a);
        count_launch();
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.B + KV_THREADS / 32 - 1) / (KV_THREADS / 32));
    cfg.blockDim = dim3(KV_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = a.total_rows > 0;   // only behind this call's own scatter
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kv_advance, a);
    count_launch();
    return e;
}

}  // namespace osp
