// IVF posting lists from the top-m assignment (paper Sections 4.2 and 4.3).
//
// Rule: a vector is stored with its best cluster (Section 4.2) and with further clusters of its top-m list, up to
// max_lists in all (the paper uses two), while their responsibility is strictly greater than tau (tau = 1 / K in the
// paper: a cluster is taken only if seeing the vector raised its posterior above the uniform prior, Section 4.3).
// Output: CSR lists, offsets[K + 1] and the vectors of each list in ascending order.  Integer work, deterministic.
//
// The N vectors are cut into at most PL_MAX_BLOCKS contiguous ranges, one CTA each, so that the scratch (one counter per
// range and cluster) does not grow with N:
//   1. pl_count_kernel: entries per (range, cluster), counted in shared memory;
//   2. pl_scan_kernel: list lengths and, per cluster, where every range starts inside the list (32 clusters per CTA, the
//      ranges split over 32 warps, so that nobody walks the ranges alone);
//   3. pl_offsets_kernel: prefix sum of the list lengths;
//   4. pl_fill_kernel: the ranges again; every WARP owns a contiguous part of its CTA's range with cursors of its own (a
//      first pass over the part counts), takes 32 vectors at a time, and ranks the entries of one list by a 32-bit map of
//      the lanes that hold it: ascending lists without a sort and without atomics on the output, all warps at work.
// 160 MB in, 60 MB out for 10M vectors with top-2 input (34 us of memory traffic).  Bound by the fill kernel's chains of
// shared-memory operations (map, cursor, map) at 24 warps per SM.  Measured at that size, K = 1024: 4.05 ms while the warps
// of a CTA filled one after the other and one thread per cluster walked the ranges; 0.30 ms now (fill 0.21, count 0.05).
#include "internal.cuh"

namespace fg {

namespace {

constexpr int PL_THREADS = 256;
constexpr int PL_MAX_LISTS = GMM_MAX_TOPM;      // at most this many lists per vector

__device__ __forceinline__ bool pl_take(int j, float r, float tau) { return j == 0 || r > tau; }

__global__ void __launch_bounds__(PL_THREADS)
pl_count_kernel(const int32_t* __restrict__ idx, const float* __restrict__ resp, int64_t n, int m, int K, float tau,
                int max_lists, int64_t range, int32_t* __restrict__ counts /* [blocks][K] */) {
    extern __shared__ int32_t hist[];
    for (int k = threadIdx.x; k < K; k += PL_THREADS) hist[k] = 0;
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * range;
    const int64_t i1 = (i0 + range < n) ? (i0 + range) : n;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += PL_THREADS) {
        for (int j = 0; j < max_lists; ++j) {
            const int32_t k = __ldg(idx + i * m + j);
            if (k < 0 || k >= K || !pl_take(j, __ldg(resp + i * m + j), tau)) break;
            atomicAdd(&hist[k], 1);                 // integer counts: the order of the additions does not matter
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += PL_THREADS) counts[(size_t)blockIdx.x * K + k] = hist[k];
}

// counts[b][k] -> where range b starts inside list k (in place; int32 is enough: a list holds fewer than 2^31 vectors);
// totals[k] = length of list k.  One CTA per 32 clusters: lane = cluster, warp w takes the w-th part of the ranges.
__global__ void __launch_bounds__(1024) pl_scan_kernel(int32_t* __restrict__ counts, int blocks, int K, int32_t* __restrict__ totals) {
    __shared__ int32_t part[32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    const int per = (blocks + 31) / 32;
    const int b0 = w * per, b1 = min(blocks, b0 + per);
    int32_t s = 0;
    if (k < K) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) s += counts[(size_t)b * K + k];
    }
    part[w][lane] = s;
    __syncthreads();
    int32_t run = 0, total = 0;
    for (int j = 0; j < 32; ++j) {
        if (j < w) run += part[j][lane];
        total += part[j][lane];
    }
    if (k >= K) return;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
        const int32_t c = counts[(size_t)b * K + k];
        counts[(size_t)b * K + k] = run;
        run += c;
    }
    if (w == 0) totals[k] = total;
}

// offsets = exclusive prefix sum of totals (one CTA of 1024 threads, 1024 clusters at a time)
__global__ void __launch_bounds__(1024) pl_offsets_kernel(const int32_t* __restrict__ totals, int K, int64_t* __restrict__ offsets) {
    __shared__ int64_t wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t carry = 0;
    for (int base = 0; base < K; base += 1024) {
        const int k = base + threadIdx.x;
        const int64_t v = (k < K) ? totals[k] : 0;
        int64_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        int64_t before = carry, total = 0;
        for (int j = 0; j < 32; ++j) {
            if (j < w) before += wsum[j];
            total += wsum[j];
        }
        if (k < K) offsets[k] = before + inc - v;
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) offsets[K] = carry;
}

// A vector's entries: the number of leading choices that pass the rule, and their clusters.  ML >= max_lists.
template <int ML>
struct PlEntries {
    int32_t k[ML];
    float r[ML];
    __device__ __forceinline__ void load(const int32_t* __restrict__ idx, const float* __restrict__ resp, int64_t i, bool in, int m, int max_lists) {
        if (ML == 2 && m == 2 && max_lists == 2) {                 // (the arrays' rows are 8 bytes; see launch_posting_lists)
            int2 a = make_int2(-1, -1);
            float2 b = make_float2(0.f, 0.f);
            if (in) { a = __ldg(reinterpret_cast<const int2*>(idx) + i); b = __ldg(reinterpret_cast<const float2*>(resp) + i); }
            k[0] = a.x; k[1] = a.y; r[0] = b.x; r[1] = b.y;
            return;
        }
#pragma unroll
        for (int j = 0; j < ML; ++j) {
            k[j] = -1;
            r[j] = 0.f;
            if (in && j < max_lists) { k[j] = __ldg(idx + i * m + j); if (j > 0) r[j] = __ldg(resp + i * m + j); }
        }
    }
    __device__ __forceinline__ int count(int K, float tau) const {
        int c = 0;
#pragma unroll
        for (int j = 0; j < ML; ++j)
            if (c == j && k[j] >= 0 && k[j] < K && pl_take(j, r[j], tau)) c = j + 1;
        return c;
    }
};

// Shared memory: cursor [W][K], lanes [W][K] (which lanes of the warp's 32 vectors hold an entry of the list; zero between
// steps).  W = blockDim.x / 32 warps.  The next step's loads are in flight while a step is placed.
template <int ML>
__global__ void __launch_bounds__(PL_THREADS)
pl_fill_kernel(const int32_t* __restrict__ idx, const float* __restrict__ resp, int64_t n, int m, int K, float tau,
               int max_lists, int64_t range, const int32_t* __restrict__ starts /* [blocks][K] */,
               const int64_t* __restrict__ offsets, int32_t* __restrict__ items) {
    extern __shared__ int32_t smem[];
    const int W = blockDim.x >> 5, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t* cursor = smem + (size_t)warp * K;
    unsigned* lanes = reinterpret_cast<unsigned*>(smem) + (size_t)(W + warp) * K;
    for (int k = tid; k < 2 * W * K; k += blockDim.x) smem[k] = 0;
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * range;
    const int64_t i1 = (i0 + range < n) ? (i0 + range) : n;
    const int64_t part = ((i1 - i0 + W - 1) / W + 31) / 32 * 32;          // this warp's vectors: [p0, p1)
    const int64_t p0 = min(i1, i0 + warp * part), p1 = min(i1, p0 + part);
    // first pass: the warp's entries per list
    for (int64_t i = p0 + lane; i < p1; i += 128) {
        PlEntries<ML> e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) e[u].load(idx, resp, i + 32 * u, i + 32 * u < p1, m, max_lists);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = e[u].count(K, tau);
#pragma unroll
            for (int j = 0; j < ML; ++j)
                if (j < c) atomicAdd(&cursor[e[u].k[j]], 1);
        }
    }
    __syncthreads();
    // where each warp starts inside every list
    for (int k = tid; k < K; k += blockDim.x) {
        int32_t c = starts[(size_t)blockIdx.x * K + k];
        for (int w = 0; w < W; ++w) {
            const int32_t cnt = smem[(size_t)w * K + k];
            smem[(size_t)w * K + k] = c;
            c += cnt;
        }
    }
    __syncthreads();
    PlEntries<ML> cur, nxt;
    cur.load(idx, resp, p0 + lane, p0 + lane < p1, m, max_lists);
    const unsigned below = (1u << lane) - 1u;
    for (int64_t base = p0; base < p1; base += 32) {
        const int64_t i = base + lane;
        nxt.load(idx, resp, i + 32, i + 32 < p1, m, max_lists);
        const int c = cur.count(K, tau);
        bool twice = false;
#pragma unroll
        for (int j = 1; j < ML; ++j)
#pragma unroll
            for (int q = 0; q < j; ++q) twice |= j < c && cur.k[q] == cur.k[j];
        if (ML > 1 && __any_sync(0xffffffffu, twice)) {
            // A row that names a cluster twice is listed there twice (the counts have it so): a bit per lane is not enough, so every
            // entry counts the others of its list, one lane of the warp after the other.
            int rank[ML], all[ML];
#pragma unroll
            for (int j = 0; j < ML; ++j) rank[j] = all[j] = 0;
            for (int src = 0; src < 32; ++src) {
#pragma unroll
                for (int q = 0; q < ML; ++q) {
                    const int32_t v = __shfl_sync(0xffffffffu, q < c ? cur.k[q] : -1, src);
#pragma unroll
                    for (int j = 0; j < ML; ++j)
                        if (j < c && cur.k[j] == v) {
                            ++all[j];
                            if (src < lane || (src == lane && q < j)) ++rank[j];
                        }
                }
            }
#pragma unroll
            for (int j = 0; j < ML; ++j)
                if (j < c) items[__ldg(offsets + cur.k[j]) + cursor[cur.k[j]] + rank[j]] = (int32_t)i;
            __syncwarp();
#pragma unroll
            for (int j = 0; j < ML; ++j)
                if (j < c && rank[j] == 0) cursor[cur.k[j]] += all[j];
            __syncwarp();
            cur = nxt;
            continue;
        }
        int64_t off[ML];
#pragma unroll
        for (int j = 0; j < ML; ++j)
            if (j < c) {
                off[j] = __ldg(offsets + cur.k[j]);
                atomicOr(&lanes[cur.k[j]], 1u << lane);
            }
        __syncwarp();
        // An entry's place inside its list: after the entries of the same list from LOWER lanes, whichever of their choices
        // it is (a first choice of vector i + 5 must not land before a second choice of i + 3).
        unsigned mk[ML];
#pragma unroll
        for (int j = 0; j < ML; ++j) {
            mk[j] = 0u;
            if (j < c) {
                mk[j] = lanes[cur.k[j]];
                items[off[j] + cursor[cur.k[j]] + __popc(mk[j] & below)] = (int32_t)i;
            }
        }
        __syncwarp();
        // the lowest lane of every list moves its cursor past the step's entries and clears the map
#pragma unroll
        for (int j = 0; j < ML; ++j)
            if (j < c && (mk[j] & below) == 0u) {
                cursor[cur.k[j]] += __popc(mk[j]);
                lanes[cur.k[j]] = 0u;
            }
        __syncwarp();
        cur = nxt;
    }
}

}  // namespace

int pl_blocks(int64_t n, int64_t* range_out) {
    int64_t range = (n + PL_MAX_BLOCKS - 1) / PL_MAX_BLOCKS;
    range = (range + PL_THREADS - 1) / PL_THREADS * PL_THREADS;        // whole steps of 256 vectors
    if (range < PL_THREADS) range = PL_THREADS;
    *range_out = range;
    return (int)((n + range - 1) / range);
}

size_t pl_scratch_bytes(int K) { return (size_t)(PL_MAX_BLOCKS + 1) * K * sizeof(int32_t); }

cudaError_t launch_posting_lists(cudaStream_t s, const int32_t* idx, const float* resp, int64_t n, int m, int K, float tau,
                                 int max_lists, void* scratch, int64_t* offsets, int32_t* items) {
    int64_t range = 0;
    const int blocks = pl_blocks(n, &range);
    int32_t* counts = static_cast<int32_t*>(scratch);
    int32_t* totals = counts + (size_t)PL_MAX_BLOCKS * K;
    const size_t smem = (size_t)K * sizeof(int32_t);
    constexpr size_t FILL_CURSORS = 100 * 1024, FILL_MOST = 3 * (size_t)PL_MAX_K * 8;
    static_assert(FILL_MOST >= FILL_CURSORS, "shared memory of the fill");
    // 8 bytes per warp and cluster: eight warps up to K = 1024 (three CTAs per SM), fewer beyond, down to three at K = 8192
    int warps = PL_THREADS / 32;
    while (warps > 3 && (size_t)warps * K * 8 > FILL_CURSORS) --warps;
    const size_t smem_fill = (size_t)warps * K * 8;
    // (two choices per vector, the paper's rule, read as 8-byte rows where the arrays allow it)
    const bool pairs = m == 2 && max_lists == 2 && (reinterpret_cast<uintptr_t>(idx) & 7) == 0 && (reinterpret_cast<uintptr_t>(resp) & 7) == 0;
    auto fill = max_lists == 1 ? pl_fill_kernel<1> : pairs ? pl_fill_kernel<2> : pl_fill_kernel<PL_MAX_LISTS>;
    // (the same limits from every call: they belong to the kernels, which contexts on other threads launch for other K)
    cudaError_t e = cudaFuncSetAttribute(pl_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PL_MAX_K * (int)sizeof(int32_t));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FILL_MOST);
    if (e != cudaSuccess) return e;
    pl_count_kernel<<<blocks, PL_THREADS, smem, s>>>(idx, resp, n, m, K, tau, max_lists, range, counts);
    pl_scan_kernel<<<(K + 31) / 32, 1024, 0, s>>>(counts, blocks, K, totals);
    pl_offsets_kernel<<<1, 1024, 0, s>>>(totals, K, offsets);
    fill<<<blocks, warps * 32, smem_fill, s>>>(idx, resp, n, m, K, tau, max_lists, range, counts, offsets, items);
    return cudaGetLastError();
}

}  // namespace fg
