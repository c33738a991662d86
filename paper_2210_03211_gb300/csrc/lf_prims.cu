// Device primitives: exclusive prefix sum and a stable LSD radix sort of
// 64-bit keys with optional 32-bit payloads.  Hand-written for sm_103a; used
// by the CSR build, the node order and the community output.
#include "lf_internal.cuh"

namespace lf {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
constexpr int64_t SCAN_DIRECT = 512;   // block sums that every block adds up itself

template <typename T>
__device__ T block_exclusive_scan(T v, T *warp_sums, T &block_total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        T s = lane < SCAN_THREADS / 32 ? warp_sums[lane] : T(0);
#pragma unroll
        for (int o = 1; o < SCAN_THREADS / 32; o <<= 1) {
            T y = __shfl_up_sync(FULL, s, o);
            if (lane >= o) s += y;
        }
        if (lane < SCAN_THREADS / 32) warp_sums[lane] = s;
    }
    __syncthreads();
    T prefix = w > 0 ? warp_sums[w - 1] : T(0);
    block_total = warp_sums[SCAN_THREADS / 32 - 1];
    __syncthreads();
    return prefix + x - v;
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(const T *in, int64_t count, T *sums) {
    __shared__ T ws[SCAN_THREADS / 32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i)
        if (base + i < count) s += in[base + i];
    T tot;
    block_exclusive_scan<T>(s, ws, tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_down(const T *in, T *out, int64_t count,
                                                            const T *block_offsets, bool sums, T *d_total) {
    __shared__ T ws[SCAN_THREADS / 32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T vals[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        vals[i] = base + i < count ? in[base + i] : T(0);
        s += vals[i];
    }
    T tot;
    T run = block_exclusive_scan<T>(s, ws, tot);
    T boff = T(0);
    if (block_offsets && sums) {   // the sums themselves: the blocks before this one are added up here
        T mine = T(0);
        for (unsigned i = threadIdx.x; i < blockIdx.x; i += SCAN_THREADS) mine += block_offsets[i];
        block_exclusive_scan<T>(mine, ws, boff);
    } else if (block_offsets) {
        boff = block_offsets[blockIdx.x];
    }
    run += boff;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < count) out[base + i] = run;
        run += vals[i];
    }
    if (d_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *d_total = boff + tot;
}

}  // namespace

template <typename T>
void scan_exclusive(lf_graph *g, const T *in, T *out, int64_t count, T *d_total) {
    if (count <= 0) {
        if (d_total) LF_CUDA(cudaMemsetAsync(d_total, 0, sizeof(T), g->stream));
        return;
    }
    int64_t nb = (count + SCAN_TILE - 1) / SCAN_TILE;
    if (nb > 0x7fffffff) fail(LF_ERR_CAPACITY, "scan of %lld elements", (long long)count);
    if (nb == 1) {
        k_scan_down<T><<<1, SCAN_THREADS, 0, g->stream>>>(in, out, count, nullptr, false, d_total);
        LF_LAUNCHED();
        g->launches += 1;
        return;
    }
    T *sums = dalloc_n<T>(g, nb);
    k_scan_reduce<T><<<(unsigned)nb, SCAN_THREADS, 0, g->stream>>>(in, count, sums);
    LF_LAUNCHED();
    // up to a few hundred sums are added up by every block for itself: a launch less
    const bool direct = nb <= SCAN_DIRECT;
    if (!direct) scan_exclusive<T>(g, sums, sums, nb, nullptr);
    k_scan_down<T><<<(unsigned)nb, SCAN_THREADS, 0, g->stream>>>(in, out, count, sums, direct, d_total);
    LF_LAUNCHED();
    g->launches += 2;
    dfree(g, sums);
}

template void scan_exclusive<int32_t>(lf_graph *, const int32_t *, int32_t *, int64_t, int32_t *);
template void scan_exclusive<uint32_t>(lf_graph *, const uint32_t *, uint32_t *, int64_t, uint32_t *);
template void scan_exclusive<int64_t>(lf_graph *, const int64_t *, int64_t *, int64_t, int64_t *);
template void scan_exclusive<unsigned long long>(lf_graph *, const unsigned long long *,
                                                 unsigned long long *, int64_t, unsigned long long *);

// ---------------------------------------------------------------------------
// LSD radix sort, 8-bit digits.  Per pass: block digit histograms (digit-major
// so that one exclusive scan gives every block its output offset per digit),
// then a stable scatter.  Each warp owns a contiguous sub-tile; inside it,
// equal digits in a 32-item chunk are grouped with __match_any_sync, so the
// rank of an item is (warp's running count for the digit) + (lanes below it
// with the same digit).  Warps, chunks and lanes are visited in input order,
// which keeps the sort stable.
//
// Bound by memory: the tile is first put in order in shared memory, then written
// digit by digit, so a block writes runs of (tile / 256) keys to neighbouring
// addresses.  Written straight from the registers, the 8 keys a digit of a 2,048-key
// tile went out one sector each and the pass ran at a seventh of the copy rate
// (230M keys, 3.7 GB: 6.3 ms -> 2.5 ms a scatter).  Tiles of 8,192 keys where
// that leaves every SM two blocks, else 2,048.
// ---------------------------------------------------------------------------
namespace {

constexpr int RS_WARPS = 16;
constexpr int RS_THREADS = RS_WARPS * 32;
constexpr int RS_ITEMS_LARGE = 16, RS_ITEMS_SMALL = 4;   // keys per thread
constexpr int64_t RS_LARGE = 2ll * 152 * RS_THREADS * RS_ITEMS_LARGE;   // keys from which large tiles are used

constexpr size_t rs_smem(int items) { return (size_t)RS_THREADS * items * 8 + (size_t)RS_WARPS * 256 * 4 + 2 * 256 * 4; }

template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const unsigned long long *keys, int64_t count,
                                                        int shift, uint32_t *counts, int nb) {
    __shared__ uint32_t h[256];
    for (int i = threadIdx.x; i < 256; i += RS_THREADS) h[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (RS_THREADS * ITEMS);
    unsigned long long k[ITEMS];
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const int64_t idx = base + c * RS_THREADS + threadIdx.x;
        k[c] = idx < count ? keys[idx] : 0ull;
    }
#pragma unroll
    for (int c = 0; c < ITEMS; ++c)
        if (base + c * RS_THREADS + threadIdx.x < count) atomicAdd(&h[(k[c] >> shift) & 255u], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += RS_THREADS) counts[(int64_t)i * nb + blockIdx.x] = h[i];
}

template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS, 2) k_rs_scatter(const unsigned long long *kin, const uint32_t *vin,
                                                              unsigned long long *kout, uint32_t *vout,
                                                              int64_t count, int shift, const uint32_t *offs,
                                                              int nb) {
    extern __shared__ unsigned long long rs_dyn[];
    constexpr int TILE = RS_THREADS * ITEMS;
    unsigned long long *s_k = rs_dyn;                                    // the tile, in order
    uint32_t (*wh)[256] = reinterpret_cast<uint32_t (*)[256]>(s_k + TILE);   // per warp: count, then place of a digit
    uint32_t *s_go = &wh[RS_WARPS][0];                                   // digit: output offset - place in the tile
    uint32_t *s_ws = s_go + 256;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < RS_WARPS * 256; i += RS_THREADS) wh[i >> 8][i & 255] = 0;
    __syncthreads();
    const int64_t tile = (int64_t)blockIdx.x * TILE;
    const int64_t base = tile + (int64_t)w * (32 * ITEMS);
    const int held = (int)(count - tile < TILE ? count - tile : TILE);
    unsigned long long k[ITEMS];
    uint16_t rank[ITEMS];
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const int64_t idx = base + c * 32 + lane;
        k[c] = idx < count ? kin[idx] : 0ull;
    }
    const unsigned lt = lanemask_lt();
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const bool valid = base + c * 32 + lane < count;
        const int dg = valid ? (int)((k[c] >> shift) & 255u) : 256 + lane;
        const unsigned mask = __match_any_sync(FULL, dg);
        rank[c] = valid ? (uint16_t)(wh[w][dg] + __popc(mask & lt)) : 0;
        __syncwarp();
        if (valid && lane == __ffs(mask) - 1) wh[w][dg] += __popc(mask);
        __syncwarp();
    }
    __syncthreads();
    {   // places of the digits in the tile: 256 totals scanned by eight warps, then the warps' shares
        const int d = threadIdx.x & 255;
        uint32_t total = 0;
        if (threadIdx.x < 256) {
#pragma unroll
            for (int ww = 0; ww < RS_WARPS; ++ww) total += wh[ww][d];
        }
        uint32_t inc = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += t;
        }
        if (threadIdx.x < 256 && lane == 31) s_ws[w] = inc;
        __syncthreads();
        if (threadIdx.x < 256) {
            uint32_t run = inc - total;
            for (int ww = 0; ww < w; ++ww) run += s_ws[ww];
            s_go[d] = offs[(int64_t)d * nb + blockIdx.x] - run;
#pragma unroll
            for (int ww = 0; ww < RS_WARPS; ++ww) {
                const uint32_t t = wh[ww][d];
                wh[ww][d] = run;
                run += t;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < ITEMS; ++c)
        if (base + c * 32 + lane < count) {
            rank[c] = (uint16_t)(rank[c] + wh[w][(k[c] >> shift) & 255u]);   // place in the tile
            s_k[rank[c]] = k[c];
        }
    __syncthreads();
    uint32_t dst[ITEMS];
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const int i = c * RS_THREADS + threadIdx.x;
        if (i < held) {
            const unsigned long long key = s_k[i];
            dst[c] = s_go[(key >> shift) & 255u] + (uint32_t)i;
            kout[dst[c]] = key;
        }
    }
    if (!vout) return;
    __syncthreads();
    uint32_t *s_v = reinterpret_cast<uint32_t *>(s_k);
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const int64_t idx = base + c * 32 + lane;
        if (idx < count) s_v[rank[c]] = vin[idx];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < ITEMS; ++c) {
        const int i = c * RS_THREADS + threadIdx.x;
        if (i < held) vout[dst[c]] = s_v[i];
    }
}

template <int ITEMS>
void rs_pass(lf_graph *g, const unsigned long long *ka, const uint32_t *va, unsigned long long *kb, uint32_t *vb,
             int64_t count, int shift, uint32_t *counts, int nb) {
    k_rs_hist<ITEMS><<<nb, RS_THREADS, 0, g->stream>>>(ka, count, shift, counts, nb);
    LF_LAUNCHED();
    scan_exclusive<uint32_t>(g, counts, counts, (int64_t)256 * nb, nullptr);
    k_rs_scatter<ITEMS><<<nb, RS_THREADS, rs_smem(ITEMS), g->stream>>>(ka, va, kb, vb, count, shift, counts, nb);
    LF_LAUNCHED();
    g->launches += 2;
}

}  // namespace

int bits_for(unsigned long long max_value) {
    int b = 0;
    while (b < 64 && (max_value >> b) != 0ull) ++b;
    return b;
}

void radix_sort(lf_graph *g, unsigned long long *keys, uint32_t *vals, int64_t count,
                const std::vector<int> &shifts) {
    if (count <= 1 || shifts.empty()) return;
    if (count > 0xffffffffll) fail(LF_ERR_CAPACITY, "radix sort of %lld keys", (long long)count);
    const bool large = count >= RS_LARGE;
    const int64_t tile = (int64_t)RS_THREADS * (large ? RS_ITEMS_LARGE : RS_ITEMS_SMALL);
    const int nb = (int)((count + tile - 1) / tile);
    if (large)
        LF_CUDA(cudaFuncSetAttribute(k_rs_scatter<RS_ITEMS_LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)rs_smem(RS_ITEMS_LARGE)));
    unsigned long long *k2 = dalloc_n<unsigned long long>(g, count);
    uint32_t *v2 = vals ? dalloc_n<uint32_t>(g, count) : nullptr;
    uint32_t *counts = dalloc_n<uint32_t>(g, (int64_t)256 * nb);
    unsigned long long *ka = keys, *kb = k2;
    uint32_t *va = vals, *vb = v2;
    for (int shift : shifts) {
        if (large) rs_pass<RS_ITEMS_LARGE>(g, ka, va, kb, vb, count, shift, counts, nb);
        else rs_pass<RS_ITEMS_SMALL>(g, ka, va, kb, vb, count, shift, counts, nb);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    if (ka != keys) {
        LF_CUDA(cudaMemcpyAsync(keys, ka, (size_t)count * sizeof(unsigned long long),
                                cudaMemcpyDeviceToDevice, g->stream));
        if (vals)
            LF_CUDA(cudaMemcpyAsync(vals, va, (size_t)count * sizeof(uint32_t), cudaMemcpyDeviceToDevice,
                                    g->stream));
    }
    dfree(g, counts);
    if (v2) dfree(g, v2);
    dfree(g, k2);
}

}  // namespace lf
