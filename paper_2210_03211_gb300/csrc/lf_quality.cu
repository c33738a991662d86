// Quality: the F1-score of a detected cover against a reference cover
// (Methods, Evaluation Criteria, F1-Score for Overlapping Communities): the
// mean over detected communities C' of max over reference communities C of
// F1(C', C) = 2 (p r) / (p + r), p = |C & C'| / |C'|, r = |C & C'| / |C|,
// 0 when they share no node.  Per detected community one warp (a block for the
// large ones) counts |C & C'| for every reference community its members belong
// to, in a shared hash table (several passes over hash parts when there are more
// candidates than the table holds); the mean is an exact sum.
#include <vector>

#include "lf_internal.cuh"

namespace lf {
namespace {

constexpr int F1_THREADS = 256;
constexpr uint32_t F1_SLOTS = 4096;

// reference memberships as (node << 32 | community)
__global__ void k_ref_keys(const int64_t *off, const int32_t *mem, int64_t kb, int64_t eb,
                           unsigned long long *keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < eb; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = kb - 1;   // community of entry i: last c with off[c] <= i
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (off[mid] <= i) lo = mid; else hi = mid - 1;
        }
        keys[i] = ((unsigned long long)(uint32_t)mem[i] << 32) | (unsigned long long)lo;
    }
}

__device__ __forceinline__ int64_t first_key(const unsigned long long *keys, int64_t eb, uint32_t node) {
    const unsigned long long k = (unsigned long long)node << 32;
    int64_t lo = 0, hi = eb;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (keys[mid] < k) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ double f1_pair(int64_t k, int64_t a, int64_t b) {
    if (k == 0) return 0.0;
    const double p = __ddiv_rn((double)k, (double)a), r = __ddiv_rn((double)k, (double)b);
    return __dmul_rn(2.0, __ddiv_rn(__dmul_rn(p, r), __dadd_rn(p, r)));
}

// (score descending, reference index ascending); c < 0 = none
__device__ __forceinline__ bool f1_better(double f1, int32_t c1, double f2, int32_t c2) {
    if (c1 < 0) return false;
    if (c2 < 0) return true;
    return f1 > f2 || (f1 == f2 && c1 < c2);
}

// Where each node's reference memberships lie in the sorted keys: [x, y) per id,
// (0, 0) for an id without any (the array starts zeroed).
__global__ void k_ref_ranges(const unsigned long long *keys, int64_t eb, uint2 *range) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < eb; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t x = (uint32_t)(keys[i] >> 32);
        if (i == 0 || (uint32_t)(keys[i - 1] >> 32) != x) range[x].x = (uint32_t)i;
        if (i + 1 == eb || (uint32_t)(keys[i + 1] >> 32) != x) range[x].y = (uint32_t)(i + 1);
    }
}

struct RefIndex {
    const unsigned long long *keys;   // (node << 32 | community), sorted
    int64_t eb;
    const uint2 *range;               // per id, or null: ids too sparse for a table, searched
    __device__ __forceinline__ void find(uint32_t x, int64_t &lo, int64_t &hi) const {
        if (range) {
            const uint2 r = range[x];
            lo = r.x;
            hi = r.y;
        } else {
            lo = first_key(keys, eb, x);
            hi = x == 0xffffffffu ? eb : first_key(keys, eb, x + 1u);
        }
    }
};

// Blocks take eight detected communities at a time, a warp each; the ones with
// more than F1_WARP_ENTRIES reference memberships are then done by the whole block, one
// after the other, so a block's eight are taken from all over the cover, and no
// block has a second one before every block has its first (8 of 100,000 members, often
// ordered by size: 94 ms with eight neighbours in one block, 12.6 ms so).
// Most communities have a dozen members: a block each cleared and scanned 4,096
// slots for them and found every member's memberships by three binary searches
// (335k nodes: 1,400 -> 540 us). A warp's table has twice as many slots as
// entries and only its used ones, listed densely, go through the FP64 divisions; a
// block's exact sum leaves it once.
constexpr uint32_t F1_WARP_SLOTS = F1_SLOTS / (F1_THREADS / 32);
constexpr uint32_t F1_WARP_ENTRIES = F1_WARP_SLOTS / 2;

__global__ void __launch_bounds__(F1_THREADS) k_cover_f1(const int64_t *off_a, const int32_t *mem_a, int64_t ka,
                                                         const int64_t *off_b, RefIndex ref, unsigned long long *sacc,
                                                         int32_t *best) {
    __shared__ int32_t hk[F1_SLOTS];
    __shared__ uint32_t hv[F1_SLOTS];
    __shared__ double s_f[F1_THREADS / 32];
    __shared__ int32_t s_c[F1_THREADS / 32];
    __shared__ unsigned long long s_bound[F1_THREADS / 32];
    __shared__ unsigned long long acc[SACC_CHUNKS];
    __shared__ uint16_t s_list[F1_THREADS / 32][F1_WARP_ENTRIES];
    __shared__ int s_over;
    constexpr int NW = F1_THREADS / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned long long *keys = ref.keys;
    for (int i = threadIdx.x; i < SACC_CHUNKS; i += F1_THREADS) acc[i] = 0ull;
    __syncthreads();
    const int64_t step = gridDim.x;   // a block's eight communities lie apart
    for (int64_t c0 = blockIdx.x; c0 < ka; c0 += step * NW) {
        if (const int64_t c = c0 + w * step; c < ka) {
            const int64_t beg = off_a[c], end = off_a[c + 1], a = end - beg;
            // candidates bound: the members' reference memberships
            unsigned long long bound = 0;
            for (int64_t i = beg + lane; i < end; i += 32) {
                int64_t lo, hi;
                ref.find((uint32_t)mem_a[i], lo, hi);
                bound += (unsigned long long)(hi - lo);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) bound += __shfl_xor_sync(FULL, bound, o);
            if (lane == 0) s_bound[w] = bound;
            if (bound <= F1_WARP_ENTRIES) {
                int32_t *tk = hk + w * F1_WARP_SLOTS;
                uint32_t *tv = hv + w * F1_WARP_SLOTS;
                uint32_t H = 32;
                while (H < 2 * (uint32_t)bound) H <<= 1;
                for (uint32_t s = lane; s < H; s += 32) {
                    tk[s] = -1;
                    tv[s] = 0u;
                }
                __syncwarp();
                for (int64_t i = beg + lane; i < end; i += 32) {
                    int64_t lo, hi;
                    ref.find((uint32_t)mem_a[i], lo, hi);
                    for (int64_t j = lo; j < hi; ++j) {
                        const int32_t cb = (int32_t)(keys[j] & 0xffffffffull);
                        uint32_t h = hash32((uint32_t)cb) & (H - 1);
                        for (uint32_t probe = 0; probe < H; ++probe) {   // at most half full
                            const int32_t prev = atomicCAS(&tk[h], -1, cb);
                            if (prev == -1 || prev == cb) {
                                atomicAdd(&tv[h], 1u);
                                break;
                            }
                            h = (h + 1) & (H - 1);
                        }
                    }
                }
                __syncwarp();
                int n = 0;
                for (uint32_t b0 = 0; b0 < H; b0 += 32) {
                    const bool used = tk[b0 + lane] >= 0;
                    const unsigned m = __ballot_sync(FULL, used);
                    if (used) s_list[w][n + __popc(m & lanemask_lt())] = (uint16_t)(b0 + lane);
                    n += __popc(m);
                }
                __syncwarp();
                double bf = 0.0;
                int32_t bc = -1;
                for (int e = lane; e < n; e += 32) {
                    const int s = s_list[w][e];
                    const int32_t cb = tk[s];
                    const double f = f1_pair(tv[s], a, off_b[cb + 1] - off_b[cb]);
                    if (f1_better(f, cb, bf, bc)) {
                        bf = f;
                        bc = cb;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const double f2 = __shfl_down_sync(FULL, bf, o);
                    const int32_t c2 = __shfl_down_sync(FULL, bc, o);
                    if (f1_better(f2, c2, bf, bc)) {
                        bf = f2;
                        bc = c2;
                    }
                }
                if (lane == 0) {
                    if (best) best[c] = bc;
                    sacc_add(acc, bc >= 0 ? bf : 0.0);
                }
            }
        }
        __syncthreads();
        for (int q = 0; q < NW && c0 + q * step < ka; ++q) {   // the large ones, the whole block
        const unsigned long long bound = s_bound[q];
        if (bound <= F1_WARP_ENTRIES) continue;
        const int64_t c = c0 + q * step;
        const int64_t beg = off_a[c], end = off_a[c + 1], a = end - beg;
        uint32_t P = bound <= F1_SLOTS / 2 ? 1u : (uint32_t)((bound + F1_SLOTS / 2 - 1) / (F1_SLOTS / 2));
        double bf = 0.0;
        int32_t bc = -1;
        for (;;) {   // a part that overflows the table makes the parts twice as many
        bf = 0.0;
        bc = -1;
        if (threadIdx.x == 0) s_over = 0;
        for (uint32_t part = 0; part < P; ++part) {
            for (uint32_t s = threadIdx.x; s < F1_SLOTS; s += F1_THREADS) {
                hk[s] = -1;
                hv[s] = 0u;
            }
            __syncthreads();
            for (int64_t i = beg + threadIdx.x; i < end; i += F1_THREADS) {
                int64_t lo, hi;
                ref.find((uint32_t)mem_a[i], lo, hi);
                for (int64_t j = lo; j < hi; ++j) {
                    const int32_t cb = (int32_t)(keys[j] & 0xffffffffull);
                    if (P > 1 && hash32((uint32_t)cb ^ 0x85ebca6bu) % P != part) continue;
                    uint32_t h = hash32((uint32_t)cb) & (F1_SLOTS - 1);
                    bool placed = false;
                    for (uint32_t probe = 0; probe < F1_SLOTS; ++probe) {
                        const int32_t prev = atomicCAS(&hk[h], -1, cb);
                        if (prev == -1 || prev == cb) {
                            atomicAdd(&hv[h], 1u);
                            placed = true;
                            break;
                        }
                        h = (h + 1) & (F1_SLOTS - 1);
                    }
                    if (!placed) s_over = 1;
                }
            }
            __syncthreads();
            for (uint32_t s = threadIdx.x; s < F1_SLOTS; s += F1_THREADS) {
                const int32_t cb = hk[s];
                if (cb < 0) continue;
                const double f = f1_pair(hv[s], a, off_b[cb + 1] - off_b[cb]);
                if (f1_better(f, cb, bf, bc)) {
                    bf = f;
                    bc = cb;
                }
            }
            __syncthreads();
        }
        if (!s_over) break;
        __syncthreads();
        P *= 2;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double f2 = __shfl_down_sync(FULL, bf, o);
            const int32_t c2 = __shfl_down_sync(FULL, bc, o);
            if (f1_better(f2, c2, bf, bc)) {
                bf = f2;
                bc = c2;
            }
        }
        if (lane == 0) {
            s_f[w] = bf;
            s_c[w] = bc;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < F1_THREADS / 32; ++k)
                if (f1_better(s_f[k], s_c[k], bf, bc)) {
                    bf = s_f[k];
                    bc = s_c[k];
                }
            if (best) best[c] = bc;
            sacc_add(acc, bc >= 0 ? bf : 0.0);
        }
        __syncthreads();
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < SACC_CHUNKS; i += F1_THREADS)
        if (acc[i]) atomicAdd(&sacc[i], acc[i]);
}

__global__ void k_f1_final(unsigned long long *sacc, int64_t ka, double *out) {
    __shared__ unsigned long long acc[SACC_CHUNKS];
    const double s = sacc_take_warp(sacc, acc);   // one warp
    if (threadIdx.x == 0) *out = ka > 0 ? __ddiv_rn(s, (double)ka) : 0.0;
}

}  // namespace
}  // namespace lf

extern "C" lf_status lf_cover_f1(const int64_t *det_offsets, const int32_t *det_members, int64_t num_det,
                                 const int64_t *ref_offsets, const int32_t *ref_members, int64_t num_ref,
                                 double *f1, int32_t *best, void *stream) {
    using namespace lf;
    if (!f1 || num_det < 0 || num_ref < 0 || (num_det > 0 && !det_offsets) || (num_ref > 0 && !ref_offsets)) {
        set_error(LF_ERR_INVALID, "invalid argument");
        return LF_ERR_INVALID;
    }
    *f1 = 0.0;
    if (num_det == 0) return LF_OK;
    lf_graph tmp;   // allocation and launch bookkeeping for the call
    tmp.stream = static_cast<cudaStream_t>(stream);
    bool own = false;
    std::vector<void *> bufs;
    lf_status rc = LF_OK;
    try {
        if (!tmp.stream) {
            LF_CUDA(cudaStreamCreateWithFlags(&tmp.stream, cudaStreamNonBlocking));
            own = true;
        }
        cudaStream_t st = tmp.stream;
        const int64_t ea = det_offsets[num_det], eb = num_ref > 0 ? ref_offsets[num_ref] : 0;
        if (det_offsets[0] != 0 || (num_ref > 0 && ref_offsets[0] != 0)) fail(LF_ERR_INVALID, "offsets must start at 0");
        if ((ea > 0 && !det_members) || (eb > 0 && !ref_members)) fail(LF_ERR_INVALID, "members is NULL");
        // whole passes without a branch (they vectorise); what is wrong is looked up afterwards
        auto offsets_ok = [](const int64_t *off, int64_t k) {
            bool ok = true;
            for (int64_t c = 0; c < k; ++c) ok &= off[c + 1] > off[c];
            return ok;
        };
        auto first_empty = [](const int64_t *off) {
            int64_t c = 0;
            while (off[c + 1] > off[c]) ++c;
            return (long long)c;
        };
        if (!offsets_ok(det_offsets, num_det))
            fail(LF_ERR_INVALID, "detected community %lld is empty", first_empty(det_offsets));
        if (!offsets_ok(ref_offsets, num_ref))
            fail(LF_ERR_INVALID, "reference community %lld is empty", first_empty(ref_offsets));
        auto largest = [](const int32_t *m, int64_t n) {   // as unsigned: a negative id is above every other
            uint32_t top = 0;
            for (int64_t i = 0; i < n; ++i) top = std::max(top, (uint32_t)m[i]);
            return top;
        };
        const uint32_t max_id = std::max(largest(det_members, ea), largest(ref_members, eb));
        if (max_id > 0x7fffffffu) fail(LF_ERR_INVALID, "negative node id");
        auto alloc = [&](size_t bytes) {
            void *d = dalloc(&tmp, bytes > 0 ? bytes : 8);
            bufs.push_back(d);
            return d;
        };
        auto up = [&](const void *h, size_t bytes) {   // a device copy of host data
            void *d = alloc(bytes);
            if (bytes) LF_CUDA(cudaMemcpyAsync(d, h, bytes, cudaMemcpyHostToDevice, st));
            return d;
        };
        auto *oa = static_cast<int64_t *>(up(det_offsets, (size_t)(num_det + 1) * 8));
        auto *ma = static_cast<int32_t *>(up(det_members, (size_t)ea * 4));
        auto *ob = static_cast<int64_t *>(num_ref > 0 ? up(ref_offsets, (size_t)(num_ref + 1) * 8) : alloc(8));
        auto *mb = static_cast<int32_t *>(up(ref_members, (size_t)eb * 4));
        auto *keys = static_cast<unsigned long long *>(alloc((size_t)eb * 8));
        auto *sacc = static_cast<unsigned long long *>(alloc(SACC_CHUNKS * 8));
        auto *bst = static_cast<int32_t *>(alloc((size_t)num_det * 4));
        auto *res = static_cast<double *>(alloc(8));
        LF_CUDA(cudaMemsetAsync(sacc, 0, SACC_CHUNKS * 8, st));
        if (eb > 0) {
            k_ref_keys<<<grid_for(eb, 256, 1 << 16), 256, 0, st>>>(ob, mb, num_ref, eb, keys);
            LF_LAUNCHED();
            std::vector<int> sh;
            for (int s = 0; s < bits_for((unsigned long long)(num_ref - 1)); s += 8) sh.push_back(s);
            for (int s = 0; s < bits_for((unsigned long long)max_id); s += 8) sh.push_back(32 + s);
            radix_sort(&tmp, keys, nullptr, eb, sh);
        }
        RefIndex ref{keys, eb, nullptr};
        const int64_t ids = (int64_t)max_id + 1;
        if (eb > 0 && ids <= 16 * (ea + eb) + (1 << 20)) {   // a table per id, unless the ids are far sparser than the covers
            uint2 *range = nullptr;
            try {
                range = static_cast<uint2 *>(alloc((size_t)ids * sizeof(uint2)));
            } catch (const Error &e) {   // no room: the keys are searched, which needs none
                if (e.status != LF_ERR_OOM) throw;
            }
            if (range) {
                LF_CUDA(cudaMemsetAsync(range, 0, (size_t)ids * sizeof(uint2), st));
                k_ref_ranges<<<grid_for(eb, 256, 1 << 16), 256, 0, st>>>(keys, eb, range);
                LF_LAUNCHED();
                ref.range = range;
            }
        }
        k_cover_f1<<<grid_for(num_det, 1, 152 * 5), F1_THREADS, 0, st>>>(oa, ma, num_det, ob, ref, sacc, bst);
        LF_LAUNCHED();
        k_f1_final<<<1, 32, 0, st>>>(sacc, num_det, res);
        LF_LAUNCHED();
        LF_CUDA(cudaMemcpyAsync(f1, res, 8, cudaMemcpyDeviceToHost, st));
        if (best) LF_CUDA(cudaMemcpyAsync(best, bst, (size_t)num_det * 4, cudaMemcpyDeviceToHost, st));
        LF_CUDA(cudaStreamSynchronize(st));
    } catch (const Error &e) {
        rc = e.status;
    } catch (...) {
        set_error(LF_ERR_CUDA, "unexpected internal error");
        rc = LF_ERR_CUDA;
    }
    for (void *p : bufs) dfree(&tmp, p);
    if (tmp.stream) cudaStreamSynchronize(tmp.stream);
    if (own) cudaStreamDestroy(tmp.stream);
    return rc;
}
