// IVF posting lists from the top-m assignment (paper Sections 4.2 and 4.3).
//
// Rule: a vector is stored with its best cluster (Section 4.2) and with further clusters of its top-m list, up to
// max_lists in all (the paper uses two), while their responsibility is strictly greater than tau (tau = 1 / K in the
// paper: a cluster is taken only if seeing the vector raised its posterior above the uniform prior, Section 4.3).
// Output: CSR lists, offsets[K + 1] and the vectors of each list in ascending order.  Integer work, deterministic.
//
// The N vectors are cut into at most PL_MAX_BLOCKS contiguous ranges, one CTA each (two per SM), so that the scratch (one counter per
// range and cluster) does not grow with N:
//   1. pl_count_kernel: entries per (range, cluster), counted in shared memory;
//   2. pl_scan_kernel: list lengths and, per cluster, where every range starts inside the list (32 clusters per CTA, the
//      ranges split over 32 warps, so that nobody walks the ranges alone); prefix sum of the list lengths;
//   3. pl_fill_kernel: the ranges again, a chunk of up to PL_SLOTS choices per warp at a time, sorted by cluster in shared memory and written from there.
// 160 MB in, 60 MB out for 10M vectors with top-2 input (34 us of memory traffic; the choices are read twice).
// Bound by the shared-memory operations of ranking and placing (half of the fill) and its scattered stores.  Measured at that size (us), K = 64, 1024, 4096: 255, 308,
// 593 when a warp counted its part of a range first, ranked lanes by a map per list and stored 32 entries into 32 lists; 227, 224, 399 now (count 39 of 55,
// scan and offsets 11 of 15, fill 144 of 209 at K = 1024).
#include "internal.cuh"

namespace fg {

namespace {

constexpr int PL_COUNT_THREADS = 1024;
constexpr int PL_WARPS = 16;                    // of the fill (fewer for many clusters)
constexpr int PL_SLOTS = 512;                   // choices of a warp in a chunk
constexpr int PL_LEAST = 512;                   // vectors of a range (at least)
static_assert(GMM_MAX_TOPM <= 8, "lanes per vector");

__device__ __forceinline__ bool pl_take(int j, float r, float tau) { return j == 0 || r > tau; }

// Lane = one choice of one vector, L lanes per vector (a power of two, at least max_lists), in the order of the lists: vector by vector, choice by choice.
// Its cluster if the vector is listed there, else -1: choices count up to the first that does not pass.
__device__ __forceinline__ void pl_load(const int32_t* __restrict__ idx, const float* __restrict__ resp, int64_t i, int j, bool in, int m, int max_lists, int& k, float& r) {
    k = -1;
    r = 0.f;
    if (in && j < max_lists) {
        k = __ldg(idx + i * m + j);
        if (j > 0) r = __ldg(resp + i * m + j);
    }
}
template <int L>
__device__ __forceinline__ int pl_listed(int k, float r, int j, int lane, int K, float tau) {
    const bool ok = k >= 0 && k < K && pl_take(j, r, tau);
    if (L == 1) return ok ? k : -1;
    const unsigned mask = __ballot_sync(0xffffffffu, ok) >> (lane & ~(L - 1)), upto = (2u << j) - 1u;
    return (mask & upto) == upto ? k : -1;
}

template <int L>
__global__ void __launch_bounds__(PL_COUNT_THREADS)
pl_count_kernel(const int32_t* __restrict__ idx, const float* __restrict__ resp, int64_t n, int m, int K, float tau,
                int max_lists, int64_t range, int32_t* __restrict__ counts /* [blocks][K] */, unsigned* __restrict__ ticket /* of the scan */) {
    extern __shared__ int32_t hist[];
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0u;
    for (int k = threadIdx.x; k < K; k += PL_COUNT_THREADS) hist[k] = 0;
    __syncthreads();
    constexpr int STEP = PL_COUNT_THREADS / L;                // vectors per step
    const int lane = threadIdx.x & 31, j = threadIdx.x & (L - 1);
    const int64_t i0 = (int64_t)blockIdx.x * range;
    const int64_t i1 = (i0 + range < n) ? (i0 + range) : n;
    for (int64_t i = i0 + threadIdx.x / L; i - threadIdx.x / L < i1; i += 4 * STEP) {
        int k[4];
        float r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) pl_load(idx, resp, i + u * STEP, j, i + u * STEP < i1, m, max_lists, k[u], r[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = pl_listed<L>(k[u], r[u], j, lane, K, tau);
            if (t >= 0) atomicAdd(&hist[t], 1);               // integer counts: the order of the additions does not matter
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += PL_COUNT_THREADS) counts[(size_t)blockIdx.x * K + k] = hist[k];
}

// counts[b][k] -> where range b starts inside list k (in place; int32 is enough: a list holds fewer than 2^31 vectors);
// totals[k] = length of list k.  One CTA per 32 clusters: lane = cluster, warp w takes the w-th part of the ranges.
// The last CTA to finish turns the lengths into the lists' offsets.
__global__ void __launch_bounds__(1024) pl_scan_kernel(int32_t* __restrict__ counts, int blocks, int K, int32_t* __restrict__ totals, unsigned* __restrict__ ticket,
                                                       int64_t* __restrict__ offsets) {
    __shared__ int32_t part[32][33];
    __shared__ int64_t wsum[32];
    __shared__ int last_s;
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
    if (k < K) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) {
            const int32_t c = counts[(size_t)b * K + k];
            counts[(size_t)b * K + k] = run;
            run += c;
        }
        if (w == 0) totals[k] = total;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last_s = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    int64_t carry = 0;
    for (int base = 0; base < K; base += 1024) {
        const int q = base + threadIdx.x;
        const int64_t v = (q < K) ? __ldcg(totals + q) : 0;
        int64_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        int64_t before = carry, sum = 0;
        for (int j = 0; j < 32; ++j) {
            if (j < w) before += wsum[j];
            sum += wsum[j];
        }
        if (q < K) offsets[q] = before + inc - v;
        carry += sum;
        __syncthreads();
    }
    if (threadIdx.x == 0) offsets[K] = carry;
}

// A CTA's range, chunk by chunk.  A warp takes a contiguous part of the chunk, its choices in registers, and ranks each among the warp's earlier choices of the
// same list: an atomic addition to the warp's cursor of the list; where two lanes of a step have the same list, in the order of the lanes
// (__match_any_sync in every step, or a vote per bit of the list's number, takes as long as all the rest: fill 203 and 228 us of 10M vectors, K = 1024,
// against 144).  Then every list's entries of the chunk get their places, in the order of the warps, and go through shared memory, so that
// neighbouring threads write neighbouring entries of a list.  (1024 choices per warp: 64 registers are too few for them.)
// Shared memory: cursors [W][K] of 16 bits, where a list's entries lie in the chunk [K] (16 bits), in the list (less that) [K], the chunk's entries
// [W * PL_SLOTS] (list, vector).
template <int L>
__global__ void __launch_bounds__(PL_WARPS * 32, 2)
pl_fill_kernel(const int32_t* __restrict__ idx, const float* __restrict__ resp, int64_t n, int m, int K, float tau,
               int max_lists, int64_t range, const int32_t* __restrict__ starts /* [blocks][K] */,
               const int64_t* __restrict__ offsets, int32_t* __restrict__ items) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int wsum[PL_WARPS];
    const int T = blockDim.x, W = T >> 5, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = lane & (L - 1), K2 = (K + 1) & ~1;
    int32_t* const to = reinterpret_cast<int32_t*>(smem);                               // [K2]
    uint32_t* const out = reinterpret_cast<uint32_t*>(to + K2);                         // [W * PL_SLOTS]
    uint16_t* const cursor = reinterpret_cast<uint16_t*>(out + W * PL_SLOTS);           // [W][K2]
    uint16_t* const at = cursor + (size_t)W * K2;                                       // [K2]
    uint16_t* const cur = cursor + (size_t)warp * K2;
    unsigned* const cur32 = reinterpret_cast<unsigned*>(cur);
    for (int k = tid; k < K; k += T) to[k] = starts[(size_t)blockIdx.x * K + k];
    const int lists = ((K + W - 1) / W + 31) / 32 * 32;
    constexpr int V = 32 / L, STEPS = PL_SLOTS / 32;                                    // vectors per step; steps of a warp
    const int64_t i0 = (int64_t)blockIdx.x * range;
    const int64_t i1 = (i0 + range < n) ? (i0 + range) : n;
    const int64_t most = (int64_t)W * STEPS * V, chunks = (i1 - i0 + most - 1) / most;
    const int part = (int)(((i1 - i0 + chunks * W - 1) / (chunks * W) + V - 1) / V * V);        // vectors per warp and chunk (at most STEPS * V)
    for (int64_t c0 = i0; c0 < i1; c0 += (int64_t)part * W) {
        for (int q = tid; q < W * K2 / 2; q += T) reinterpret_cast<uint32_t*>(cursor)[q] = 0u;
        const int64_t p0 = c0 + warp * part, p1 = p0 + part < i1 ? p0 + part : i1;
        int list[STEPS];                                     // the choice's list (-1: none), then also its rank
#pragma unroll
        for (int s0 = 0; s0 < STEPS; s0 += 8) {
            float r[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const int64_t i = p0 + (s0 + s) * V + lane / L;
                pl_load(idx, resp, i, j, i < p1, m, max_lists, list[s0 + s], r[s]);
            }
#pragma unroll
            for (int s = 0; s < 8; ++s) list[s0 + s] = pl_listed<L>(list[s0 + s], r[s], j, lane, K, tau);
        }
        {   // the next chunk's choices are on their way into L2
            const int64_t b = (p0 + (int64_t)part * W) * m * 4 + lane * 128, e = (p1 + (int64_t)part * W < i1 ? p1 + (int64_t)part * W : i1) * m * 4;
            for (int64_t q = b; q < e; q += 32 * 128) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(idx) + q));
                if (L > 1) asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(resp) + q));
            }
        }
        __syncthreads();                                     // (cursors are zero; the entries of the chunk before have been written)
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
            if (p0 + s * V >= p1) break;
            const int k = list[s], sh = 16 * (k & 1);
            int c = 0, now = 1;
            if (k >= 0) c = (int)((atomicAdd(cur32 + (k >> 1), 1u << sh) >> sh) & 0xffffu);
            __syncwarp();
            if (k >= 0) now = cur[k];
            // (two of this step in one list: in the order of the lanes)
            if (__any_sync(0xffffffffu, now != c + 1)) {
                const unsigned peers = __match_any_sync(0xffffffffu, k);
                c = now - __popc(peers) + __popc(peers & ((1u << lane) - 1u));
            }
            if (k >= 0) list[s] = k | (c << 16);
        }
        __syncthreads();
        // every list's place in the chunk: a warp has a part of the lists, 32 at a time
        const int k0 = min(K, warp * lists), k1 = min(K, k0 + lists);
        int own = 0;
        for (int kb = k0; kb < k1; kb += 32) {
            const int k = kb + lane;
            int c = 0;
            if (k < k1) {
#pragma unroll 4
                for (int w = 0; w < W; ++w) { const int v = cursor[(size_t)w * K2 + k]; cursor[(size_t)w * K2 + k] = (uint16_t)c; c += v; }
            }
            int inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if (k < k1) at[k] = (uint16_t)(own + inc - c);
            own += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) wsum[warp] = own;
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < W; ++w) {
            if (w < warp) before += wsum[w];
            total += wsum[w];
        }
        for (int k = k0 + lane; k < k1; k += 32) {
            const int run = at[k] + before;
            at[k] = (uint16_t)run;
            to[k] -= run;                                    // (an entry at place p of the chunk is entry to + p of its list)
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
            if (p0 + s * V >= p1) break;
            if (list[s] >= 0) {
                const int k = list[s] & 0xffff;
                out[at[k] + cur[k] + (list[s] >> 16)] = ((uint32_t)k << 16) | (uint32_t)(warp * part + s * V + lane / L);
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int p = tid; p < total; p += T) {
            const uint32_t e = out[p];
            const int k = (int)(e >> 16);
            items[__ldg(offsets + k) + (to[k] + p)] = (int32_t)(c0 + (e & 0xffffu));
        }
        __syncthreads();
        for (int k = k0 + lane; k < k1; k += 32) to[k] += k + 1 < K ? (int)at[k + 1] : total;       // (where the next chunk's entries of the list start)
    }
}

}  // namespace

// Warps of the fill by what their cursors leave room for: two CTAs per SM up to K = 4096, one beyond.
static int pl_warps(int K) { return K <= 2048 ? PL_WARPS : PL_WARPS / 2; }

int pl_blocks(int64_t n, int64_t* range_out) {
    int64_t range = (n + PL_MAX_BLOCKS - 1) / PL_MAX_BLOCKS;
    range = (range + 255) / 256 * 256;
    if (range < PL_LEAST) range = PL_LEAST;
    *range_out = range;
    return (int)((n + range - 1) / range);
}

size_t pl_scratch_bytes(int K) { return ((size_t)(PL_MAX_BLOCKS + 1) * K + 1) * sizeof(int32_t); }      // counts, list lengths, a ticket

template <int L>
static cudaError_t launch_lists(cudaStream_t s, const int32_t* idx, const float* resp, int64_t n, int m, int K, float tau, int max_lists, int64_t range, int blocks,
                                int32_t* counts, int32_t* totals, int64_t* offsets, int32_t* items) {
    const int warps = pl_warps(K), K2 = (K + 1) & ~1;
    unsigned* ticket = reinterpret_cast<unsigned*>(totals + K);
    const size_t smem = (size_t)K2 * 4 + (size_t)warps * PL_SLOTS * 4 + (size_t)(warps + 1) * K2 * 2;
    constexpr size_t FILL_MOST = 200 * 1024;
    if (smem > FILL_MOST) return cudaErrorInvalidValue;      // (K = 8192: 192 KB)
    // (the same limits from every call: they belong to the kernels, which contexts on other threads launch for other K)
    cudaError_t e = cudaFuncSetAttribute(pl_count_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, PL_MAX_K * (int)sizeof(int32_t));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(pl_fill_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FILL_MOST);
    if (e != cudaSuccess) return e;
    pl_count_kernel<L><<<blocks, PL_COUNT_THREADS, (size_t)K * sizeof(int32_t), s>>>(idx, resp, n, m, K, tau, max_lists, range, counts, ticket);
    pl_scan_kernel<<<(K + 31) / 32, 1024, 0, s>>>(counts, blocks, K, totals, ticket, offsets);
    pl_fill_kernel<L><<<blocks, warps * 32, smem, s>>>(idx, resp, n, m, K, tau, max_lists, range, counts, offsets, items);
    return cudaGetLastError();
}

cudaError_t launch_posting_lists(cudaStream_t s, const int32_t* idx, const float* resp, int64_t n, int m, int K, float tau,
                                 int max_lists, void* scratch, int64_t* offsets, int32_t* items) {
    int64_t range = 0;
    const int blocks = pl_blocks(n, &range);
    int32_t* counts = static_cast<int32_t*>(scratch);
    int32_t* totals = counts + (size_t)PL_MAX_BLOCKS * K;
#define FG_LISTS(L_) launch_lists<L_>(s, idx, resp, n, m, K, tau, max_lists, range, blocks, counts, totals, offsets, items)
    return max_lists == 1 ? FG_LISTS(1) : max_lists == 2 ? FG_LISTS(2) : max_lists <= 4 ? FG_LISTS(4) : FG_LISTS(8);
#undef FG_LISTS
}

}  // namespace fg
