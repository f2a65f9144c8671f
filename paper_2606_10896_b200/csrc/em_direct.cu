// The FP32 path for D <= 128: direct differences on the CUDA cores, tiles cut to the shape.  (Shapes that fill the fixed tiles of
// em_fp32.cu stay there: see fp32_fixed_tiles.)
//
// log2 z = c - sum_d t^2, t = (x - g) sqrt(w2) - (mu - g) sqrt(w2) (two FMAs per term, g: a per-dimension centre near the data).  A CTA
// of 256 threads takes tiles of points.  For the logits a point belongs to G x S neighbouring lanes: G lanes own the components
// (four each, 64 per block at most), S lanes share the dimensions; a lane works on PT points at once.  For the statistics a thread
// owns a tile of TK components x 4 dimensions of the two sums, and as many replicas of those tiles as fit 256 threads split the
// points; they meet once, at the end of the kernel.  So neither K = 8 nor D = 16 pays for the 64 components x 32 (and x 128)
// dimensions that fixed tiles pad to: 10K x 16, K = 8 took 115 us per iteration with those and now takes 18 (10 us this kernel);
// 1M x 16, K = 8: 1580 -> 100 us, 1M x 96, K = 32: 2650 -> 1080 us.
//
//   DK_FUSED  K <= 64: log-sum-exp and statistics in one pass over X, the parameters stay in shared memory.
//   DK_LSE    log2 Z per point and the log-likelihood, any K (blocks of 64 components one after the other).
//   DK_STATS  statistics of a block of 64 components (blockIdx.y), given log2 Z.
//
// Bound by the FMA rate at larger K D (4 K D FMAs per point, two per instruction: fma.f32x2), by launches and the trip through X
// at small ones.
#include "internal.cuh"
#include <type_traits>
#include <math_constants.h>
#include <stdint.h>

namespace fg {

namespace {

constexpr int NT = 256;
enum { DK_FUSED = 0, DK_LSE = 1, DK_STATS = 2 };

struct DirectArgs {
    const float* X;
    int64_t n;
    int D, K;
    const float *mu, *w2;
    const double* c2d;
    const float* g;          // centre (not DK_FUSED, which takes the mean of the means itself)
    float* g_out;            // and leaves it here
    double* logZ2;           // DK_LSE writes (may be NULL), DK_STATS reads
    double* llpart;          // [gridDim.x], may be NULL
    int ll_first;            // llpart is written, not added to
    float* partials;         // [splits][K + 2 K D]
    int* status;             // DK_FUSED: parameters that are not finite and positive
    int* counts;             // DK_FUSED: zeroed for the update that follows
    const int* stop_at;      // NULL, or the iteration after which nothing is done any more
    int iter;
    int lgG, lgS;            // lanes per point: components, dimensions
    int NS;                  // a tile's points are taken in NS rounds
    int ld, ldr, kr;         // row strides (multiples of 4, odd multiples: no bank conflicts), rows of the parameters
    int D4, lgX;             // chunks of four dimensions; lanes per row when X is staged
    int T, R;                // tiles of the statistics, replicas
    int xvec;                // rows of X start on 16-byte boundaries
};

__device__ __forceinline__ float dk_ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
typedef unsigned long long u64;
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) { u64 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ u64 add2(u64 a, u64 b) { u64 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ u64 mul2(u64 a, u64 b) { u64 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ u64 dup2(float a) { u64 r; asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a)); return r; }
__device__ __forceinline__ float lo2(u64 a) { return __uint_as_float((uint32_t)a); }
__device__ __forceinline__ float hi2(u64 a) { return __uint_as_float((uint32_t)(a >> 32)); }

// The kernels of a fit follow one another at once (programmatic launch): a kernel's CTAs are started while the last ones of its
// predecessor are still at work, and wait here until those have finished and their writes are visible.  (So nothing here is read
// through the non-coherent cache.)
__device__ __forceinline__ void grid_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int MODE, int PT, int TK>
__global__ void __launch_bounds__(NT, 2) direct_kernel(const DirectArgs p) {
    extern __shared__ __align__(16) float sm[];
    grid_wait();
    const int stop = p.stop_at ? __ldcg(p.stop_at) : p.iter;      // (looked at when the first loads are under way)
    __shared__ __align__(16) float gs[128];
    __shared__ double red[NT / 32][64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int D = p.D, K = p.K, D4 = p.D4, ld = p.ld, ldr = p.ldr, kr = p.kr;
    const int lgL = p.lgG + p.lgS, G = 1 << p.lgG, S = 1 << p.lgS;
    const int s = tid & (S - 1), gq = (tid >> p.lgS) & (G - 1), pg = tid >> lgL, PG = NT >> lgL;
    const int NS = (PT == 4 && MODE != DK_LSE) ? 1 : p.NS, TP = NS * PT * PG;      // (known at compile time where registers are short)
    float* sw = sm;                          // [kr][ld] sqrt(w2)
    float* ms = sw + kr * ld;                // [kr][ld] (g - mu) sqrt(w2)
    float* xs = ms + kr * ld;                // [TP][ld] x - g
    float* rs = xs + TP * ld;                // [TP][ldr] responsibilities
    float2* run_s = reinterpret_cast<float2*>(rs);      // DK_LSE, several blocks of components: [TP] largest value, sum
    float* lz_s = rs + TP * ldr;             // DK_STATS: [TP] log2 Z
    const int kfirst = MODE == DK_STATS ? (int)blockIdx.y * 64 : 0;
    const int nblk = MODE == DK_LSE ? (K + 63) / 64 : 1;
    const int64_t ntiles = (p.n + TP - 1) / TP;

    // parameters of the block from component k0 on (raw: the means as they are)
    const int cx = tid & ((1 << p.lgX) - 1), rx = tid >> p.lgX, stepx = NT >> p.lgX;
    const bool pvec = (D & 3) == 0 && (((reinterpret_cast<uintptr_t>(p.mu) | reinterpret_cast<uintptr_t>(p.w2)) & 15) == 0);
    auto params = [&](int k0, bool raw) {
        if (cx >= D4) return;
        const int c = 4 * cx;
        const float g0 = gs[c], g1 = gs[c + 1], g2 = gs[c + 2], g3 = gs[c + 3];
#pragma unroll 4
        for (int r = rx; r < kr; r += stepx) {
            float4 m = make_float4(0.f, 0.f, 0.f, 0.f), w = m;
            if (k0 + r < K && r < 64) {
                const size_t o = (size_t)(k0 + r) * D + c;
                if (pvec) {
                    m = __ldcg(reinterpret_cast<const float4*>(p.mu + o));
                    w = __ldcg(reinterpret_cast<const float4*>(p.w2 + o));
                } else {
                    m.x = __ldcg(p.mu + o); w.x = __ldcg(p.w2 + o);
                    if (c + 1 < D) { m.y = __ldcg(p.mu + o + 1); w.y = __ldcg(p.w2 + o + 1); }
                    if (c + 2 < D) { m.z = __ldcg(p.mu + o + 2); w.z = __ldcg(p.w2 + o + 2); }
                    if (c + 3 < D) { m.w = __ldcg(p.mu + o + 3); w.w = __ldcg(p.w2 + o + 3); }
                }
                w = make_float4(sqrtf(w.x), sqrtf(w.y), sqrtf(w.z), sqrtf(w.w));
                if (!raw) m = make_float4((g0 - m.x) * w.x, (g1 - m.y) * w.y, (g2 - m.z) * w.z, (g3 - m.w) * w.w);
            }
            *reinterpret_cast<float4*>(sw + r * ld + c) = w;
            *reinterpret_cast<float4*>(ms + r * ld + c) = m;
        }
    };
    float cv[4];
    auto constants = [&](int k0) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = gq + G * b;
            cv[b] = (k0 + r < K && r < 64) ? (float)__ldcg(p.c2d + k0 + r) : -CUDART_INF_F;
        }
    };
    // a tile of X on its way into shared memory, as it is; and its arrival: a thread centres the chunks that it asked for
    auto tile_fetch = [&](int64_t row0) {
        if (cx < D4) {
            const int c = 4 * cx;
#pragma unroll 4
            for (int r = rx; r < TP; r += stepx) {
                const int64_t row = row0 + r;
                float* dst = xs + r * ld + c;
                if (row >= p.n) continue;
                const float* src = p.X + row * D + c;
                const uint32_t da = (uint32_t)__cvta_generic_to_shared(dst);
                if (p.xvec) {
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(da), "l"(src) : "memory");
                } else {
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(da), "l"(src) : "memory");
                    if (c + 1 < D) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(da + 4), "l"(src + 1) : "memory");
                    if (c + 2 < D) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(da + 8), "l"(src + 2) : "memory");
                    if (c + 3 < D) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(da + 12), "l"(src + 3) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto tile_centre = [&](int64_t row0) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (cx < D4) {
            const int c = 4 * cx;
            const float4 gv = *reinterpret_cast<const float4*>(gs + c);          // (zero beyond D)
#pragma unroll 4
            for (int r = rx; r < TP; r += stepx) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row0 + r < p.n) {
                    v = *reinterpret_cast<const float4*>(xs + r * ld + c);
                    v.x -= gv.x; v.y = c + 1 < D ? v.y - gv.y : 0.f; v.z = c + 2 < D ? v.z - gv.z : 0.f; v.w = c + 3 < D ? v.w - gv.w : 0.f;
                }
                *reinterpret_cast<float4*>(xs + r * ld + c) = v;
            }
        }
    };
    if (MODE == DK_FUSED) {
        tile_fetch((int64_t)blockIdx.x * TP);
        constants(0);
        params(0, true);                                     // (gs is not read)
        if (stop < p.iter) { asm volatile("cp.async.wait_group 0;" ::: "memory"); return; }
        if (blockIdx.x == 0 && p.counts && tid < 2) p.counts[tid] = 0;
        __syncthreads();
        int bad = 0;
        if (tid < 128) {
            double a = 0.0;
            if (tid < 4 * D4) {
#pragma unroll 4
                for (int k = 0; k < K; ++k) a += (double)ms[k * ld + tid];
            }
            const int d = tid;
            const float c = (float)(a / (double)K);
            gs[d] = isfinite(c) ? c : 0.f;
            if (blockIdx.x == 0 && p.g_out && d < D) p.g_out[d] = gs[d];
        }
        __syncthreads();
        for (int r = warp; r < K; r += NT / 32)
            for (int d = lane; d < D; d += 32) {
                const float m = ms[r * ld + d], w = sw[r * ld + d];
                if (!isfinite(m)) bad |= ST_NONFINITE;
                if (!(w > 0.f) || !isfinite(w)) bad |= ST_BAD_VAR;
                ms[r * ld + d] = (gs[d] - m) * w;
            }
        if (p.stop_at && blockIdx.x == 0 && tid < K && isnan(__ldcg(p.c2d + tid))) bad |= ST_BAD_PI;
        // (of a fit: the first iteration's parameters were checked by the preparation, the later ones here)
        if (p.stop_at && blockIdx.x == 0 && bad) atomicOr(p.status, bad);
    } else {
        tile_fetch((int64_t)blockIdx.x * TP);
        if (tid < 128) gs[tid] = (p.g && tid < D) ? __ldcg(p.g + tid) : 0.f;
        __syncthreads();
        if (nblk == 1) { params(kfirst, false); constants(kfirst); }
    }

    // statistics: thread = replica rep of tile (kt, dt)
    const int rep = tid / p.T, tt = tid - rep * p.T, dt = tt % D4, kt = tt / D4;
    u64 acc1[TK][2], acc2[TK][2];
    float nacc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < TK; ++c) acc1[c][0] = acc1[c][1] = acc2[c][0] = acc2[c][1] = 0ull;
    double ll = 0.0;

    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t row0 = t * TP;
        if (t != blockIdx.x) {
            __syncthreads();                                 // (the tile before this one has been read)
            tile_fetch(row0);
        }
        if (MODE == DK_STATS)
            for (int r = tid; r < TP; r += NT) lz_s[r] = row0 + r < p.n ? (float)__ldcg(p.logZ2 + row0 + r) : CUDART_INF_F;
        tile_centre(row0);
        __syncthreads();
        for (int blk = 0; blk < nblk; ++blk) {
            if (nblk > 1) {
                __syncthreads();
                params(blk * 64, false);
                constants(blk * 64);
                __syncthreads();
            }
#pragma unroll 1
            for (int sub = 0; sub < NS; ++sub) {
                const int p0 = sub * PT * PG + pg;           // this lane's points: p0 + j PG
                float m_run[PT], s_run[PT];
                float l[PT][4];
#pragma unroll
                for (int j = 0; j < PT; ++j) {
                    m_run[j] = -CUDART_INF_F;
                    s_run[j] = 0.f;
                    if (MODE == DK_LSE && blk > 0) { const float2 v = run_s[p0 + j * PG]; m_run[j] = v.x; s_run[j] = v.y; }
                }
                u64 q[PT][4];
#pragma unroll
                for (int j = 0; j < PT; ++j)
#pragma unroll
                    for (int b = 0; b < 4; ++b) q[j][b] = 0ull;
#pragma unroll 2
                for (int d4 = s; d4 < D4; d4 += S) {
                    ulonglong2 x[PT];
#pragma unroll
                    for (int j = 0; j < PT; ++j) x[j] = *reinterpret_cast<const ulonglong2*>(xs + (p0 + j * PG) * ld + 4 * d4);
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(sw + (gq + G * b) * ld + 4 * d4);
                        const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(ms + (gq + G * b) * ld + 4 * d4);
#pragma unroll
                        for (int j = 0; j < PT; ++j) {
                            const u64 t0 = fma2(x[j].x, w.x, m.x), t1 = fma2(x[j].y, w.y, m.y);
                            q[j][b] = fma2(t0, t0, q[j][b]);
                            q[j][b] = fma2(t1, t1, q[j][b]);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < PT; ++j) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        float v = lo2(q[j][b]) + hi2(q[j][b]);
                        for (int o = 1; o < S; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                        l[j][b] = cv[b] - v;
                    }
                    if (MODE != DK_STATS) {
                        float m = fmaxf(fmaxf(l[j][0], l[j][1]), fmaxf(l[j][2], l[j][3]));
                        for (int o = S; o < (1 << lgL); o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                        m = fmaxf(m, m_run[j]);
                        const float ref = m == -CUDART_INF_F ? 0.f : m;
                        float e[4], a;
#pragma unroll
                        for (int b = 0; b < 4; ++b) e[b] = dk_ex2(l[j][b] - ref);
                        a = (e[0] + e[1]) + (e[2] + e[3]);
                        for (int o = S; o < (1 << lgL); o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                        s_run[j] = (MODE == DK_FUSED ? 0.f : s_run[j] * dk_ex2(m_run[j] - ref)) + a;
                        m_run[j] = m;
                        if (MODE == DK_FUSED) {
#pragma unroll
                            for (int b = 0; b < 4; ++b) l[j][b] = e[b];
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < PT; ++j) {
                    const int r = p0 + j * PG;
                    const int64_t row = row0 + r;
                    const bool in = row < p.n;
                    if (MODE != DK_STATS) {
                        if (blk + 1 == nblk) {
                            const double lz = (double)m_run[j] + (double)log2f(s_run[j]);
                            if (in && (tid & ((1 << lgL) - 1)) == 0) {
                                ll += lz;
                                if (p.logZ2) p.logZ2[row] = lz;
                            }
                        } else if ((tid & ((1 << lgL) - 1)) == 0) {
                            run_s[r] = make_float2(m_run[j], s_run[j]);      // (read after the barriers of the next block)
                        }
                    }
                    if (MODE != DK_LSE) {
                        float f = 0.f, lz = 0.f;
                        if (MODE == DK_FUSED) f = in ? 1.0f / s_run[j] : 0.f;
                        else lz = lz_s[r];
                        if (s == 0) {
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                const float v = MODE == DK_FUSED ? l[j][b] * f : dk_ex2(l[j][b] - lz);
                                nacc[b] += v;
                                if (gq + G * b < ldr) rs[r * ldr + gq + G * b] = v;
                            }
                        }
                    }
                }
            }
        }
        if (MODE != DK_LSE) {
            __syncthreads();
            if (rep < p.R) {
#pragma unroll 2
                for (int r = rep; r < TP; r += p.R) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(xs + r * ld + 4 * dt);
                    const u64 y0 = mul2(x.x, x.x), y1 = mul2(x.y, x.y);
#pragma unroll
                    for (int h = 0; h < TK / 4; ++h) {
                        const float4 w = *reinterpret_cast<const float4*>(rs + r * ldr + kt * TK + 4 * h);
                        const float rr[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const u64 rd = dup2(rr[c]);
                            acc1[4 * h + c][0] = fma2(rd, x.x, acc1[4 * h + c][0]);
                            acc1[4 * h + c][1] = fma2(rd, x.y, acc1[4 * h + c][1]);
                            acc2[4 * h + c][0] = fma2(rd, y0, acc2[4 * h + c][0]);
                            acc2[4 * h + c][1] = fma2(rd, y1, acc2[4 * h + c][1]);
                        }
                    }
                }
            }
        }
    }

    // ---- once per CTA: log-likelihood, N_k, and the replicas' sums in a fixed order ----
    if (MODE != DK_STATS && p.llpart) {
        for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);
        if (lane == 0) red[warp][0] = ll;
        __syncthreads();
        if (tid == 0) {
            double a = 0.0;
            for (int w = 0; w < NT / 32; ++w) a += red[w][0];
            a *= 0.69314718055994530942;
            p.llpart[blockIdx.x] = p.ll_first ? a : p.llpart[blockIdx.x] + a;
        }
    }
    if (MODE == DK_LSE) return;
    __syncthreads();
    const size_t KD = (size_t)K * D;
    float* pN = p.partials + (size_t)blockIdx.x * (K + 2 * KD);
    float* pS1 = pN + K;
    float* pS2 = pS1 + KD;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        double a = s == 0 ? (double)nacc[b] : 0.0;
        for (int o = 16; o >= (1 << lgL); o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane < (1 << lgL) && s == 0) red[warp][gq + G * b] = a;
    }
    __syncthreads();
    if (tid < 64 && tid < 4 * G && kfirst + tid < K) {
        double a = 0.0;
        for (int w = 0; w < NT / 32; ++w) a += red[w][tid];
        pN[kfirst + tid] = (float)a;
    }
    auto put = [&](int tile, int i, float v) {               // value i of a tile: component, sum, dimension
        const int k = kfirst + (tile / D4) * TK + (i >> 3), d = (tile % D4) * 4 + (i & 3);
        if (k < K && (tile / D4) * TK + (i >> 3) < 64 && d < D) ((i & 4) ? pS2 : pS1)[(size_t)k * D + d] = v;
    };
    if (p.R == 1) {
        if (rep < 1) {
#pragma unroll
            for (int c = 0; c < TK; ++c) {
                put(tt, 8 * c, lo2(acc1[c][0])); put(tt, 8 * c + 1, hi2(acc1[c][0]));
                put(tt, 8 * c + 2, lo2(acc1[c][1])); put(tt, 8 * c + 3, hi2(acc1[c][1]));
                put(tt, 8 * c + 4, lo2(acc2[c][0])); put(tt, 8 * c + 5, hi2(acc2[c][0]));
                put(tt, 8 * c + 6, lo2(acc2[c][1])); put(tt, 8 * c + 7, hi2(acc2[c][1]));
            }
        }
        return;
    }
    float* dump = sm;                                        // [8 TK][NT + T] (no bank conflicts below), over the tiles (which all threads have left)
    const int ds = NT + p.T;
#pragma unroll
    for (int c = 0; c < TK; ++c) {
        dump[(8 * c) * ds + tid] = lo2(acc1[c][0]); dump[(8 * c + 1) * ds + tid] = hi2(acc1[c][0]);
        dump[(8 * c + 2) * ds + tid] = lo2(acc1[c][1]); dump[(8 * c + 3) * ds + tid] = hi2(acc1[c][1]);
        dump[(8 * c + 4) * ds + tid] = lo2(acc2[c][0]); dump[(8 * c + 5) * ds + tid] = hi2(acc2[c][0]);
        dump[(8 * c + 6) * ds + tid] = lo2(acc2[c][1]); dump[(8 * c + 7) * ds + tid] = hi2(acc2[c][1]);
    }
    __syncthreads();
    for (int o = tid; o < p.T * 8 * TK; o += NT) {
        const int i = o / p.T, tile = o - i * p.T;
        double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int r = 0; r < p.R; ++r) a[r & 3] += (double)dump[i * ds + r * p.T + tile];
        put(tile, i, (float)((a[0] + a[1]) + (a[2] + a[3])));
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Partials -> statistics, and in a fit the update and the next iteration's constants: a CTA per component.  Threads share the
// splits (one thread per output walked them all before: 45 us for 296 splits of K = 8, D = 16; now 6 with the update).  The sums are
// in float64, in a fixed order.
struct ReduceArgs {
    int D, K, splits;
    const float* partials;
    const float* g;
    double *Nk, *S1, *S2;
    int accumulate;
    // log-likelihood: sum of llpart[n_ll] into *ll (n_ll = 0: left alone)
    const double* llpart;
    int n_ll;
    double* ll;
    int ll_accumulate;
    // update (fit): NULL pi = none
    float *pi, *mu, *var;
    float var_floor;
    int isotropic;
    int64_t N;
    int* counts;
    const int* status;
    float* w2;
    float* c2;
    double* c2d;
    const double* ll_prev;   // NULL in the first iteration
    double tol;
    int* stop_at;
    int iter;
};

__global__ void __launch_bounds__(1024) direct_reduce_kernel(const ReduceArgs p) {
    grid_wait();
    if (p.stop_at && *p.stop_at < p.iter) return;
    __shared__ double part[1024];
    __shared__ double tot[257];
    __shared__ double red[32];
    const int tid = threadIdx.x, lane = tid & 31, k = blockIdx.x, D = p.D, W = 2 * D + 1, RG = 1024 / W;
    const size_t KD = (size_t)p.K * D, per = (size_t)p.K + 2 * KD;
    const int out = tid % W, rg = tid / W;
    double a = 0.0;
    double ll = 0.0;                                         // every CTA of a fit needs to know whether the log-likelihood is finite
    if (p.n_ll > 0 && (p.pi || k == 0) && tid < p.n_ll) ll = __ldcg(p.llpart + tid);      // (n_ll <= 1024)
    if (rg < RG) {
        const size_t e = out == 0 ? (size_t)k : out <= D ? (size_t)p.K + (size_t)k * D + out - 1 : (size_t)p.K + KD + (size_t)k * D + out - 1 - D;
        for (int r = rg; r < p.splits; r += 8 * RG) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = r + u * RG < p.splits ? __ldcg(p.partials + (size_t)(r + u * RG) * per + e) : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) a += (double)v[u];
        }
    }
    part[tid] = a;
    if (p.n_ll > 0 && (p.pi || k == 0)) {
        for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(0xffffffffu, ll, o);
        if (lane == 0) red[tid >> 5] = ll;
    }
    __syncthreads();
    if (tid < W) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int r = 0; r < RG; ++r) s[r & 3] += part[r * W + tid];
        tot[tid] = (s[0] + s[1]) + (s[2] + s[3]);
    }
    ll = 0.0;
    if (p.n_ll > 0 && (p.pi || k == 0))
        for (int w = 0; w < 32; ++w) ll += red[w];
    __syncthreads();
    // shift from the centre: S1 = S1c + g N, S2 = S2c + 2 g S1c + g^2 N
    double n = tot[0], s1 = 0.0, s2 = 0.0;
    if (tid < D) {
        const double g = p.g ? (double)__ldcg(p.g + tid) : 0.0;
        s1 = tot[1 + tid] + g * n;
        s2 = tot[1 + D + tid] + 2.0 * g * tot[1 + tid] + g * g * n;
    }
    if (p.accumulate) {
        n += p.Nk[k];
        if (tid < D) { s1 += p.S1[(size_t)k * D + tid]; s2 += p.S2[(size_t)k * D + tid]; }
    }
    __syncthreads();                                         // (everyone has read N_k)
    if (tid == 0) p.Nk[k] = n;
    if (tid < D) { p.S1[(size_t)k * D + tid] = s1; p.S2[(size_t)k * D + tid] = s2; }
    if (k == 0 && tid == 0 && p.n_ll > 0) *p.ll = p.ll_accumulate ? *p.ll + ll : ll;
    if (!p.pi) return;
    const bool good = *p.status == 0 && isfinite(ll);        // a step that failed leaves the parameters as they are
    if (k == 0 && tid == 0 && (!good || (p.tol > 0.0 && p.ll_prev && fabs(ll - *p.ll_prev) <= p.tol * fabs(ll)))) *p.stop_at = p.iter;
    if (!good) return;
    if (tid == 0) p.pi[k] = (float)(n / (double)p.N);        // pi_k = N_k / N
    const bool empty = n < 1e-12;                            // an empty component keeps mu and var
    double v = 0.0;
    float vf = 0.f;
    if (tid < D) {
        if (!empty) {
            const double m = s1 / n;                         // Eq. 2
            v = s2 / n - m * m;                              // Eq. 3 per dimension, new mean
            p.mu[(size_t)k * D + tid] = (float)m;
        }
    }
    if (empty) {
        if (tid == 0) atomicAdd(p.counts + 1, 1);
        if (tid < D) vf = p.var[(size_t)k * D + tid];
    } else {
        const double fl = (double)p.var_floor;
        if (p.isotropic) {                                   // one variance: the mean over the dimensions
            double q = tid < D ? v : 0.0;
            for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            if (lane == 0) red[tid >> 5] = q;
            __syncthreads();
            v = 0.0;
            for (int w = 0; w < 4; ++w) v += red[w];
            v /= (double)D;
            if (!(v > fl)) { v = fl; if (tid == 0) atomicAdd(p.counts, D); }
        } else if (tid < D && !(v > fl)) {
            v = fl;
            atomicAdd(p.counts, 1);
        }
        vf = (float)v;
        if (tid < D) p.var[(size_t)k * D + tid] = vf;
    }
    // the next iteration's constants
    double lg = 0.0;
    if (tid < D) {
        lg = log(6.283185307179586476925286766559 * (double)vf);
        p.w2[(size_t)k * D + tid] = (float)(0.72134752044448170368 / (double)vf);
    }
    for (int o = 16; o > 0; o >>= 1) lg += __shfl_xor_sync(0xffffffffu, lg, o);
    __syncthreads();
    if (lane == 0) red[tid >> 5] = lg;
    __syncthreads();
    if (tid == 0) {
        const float pf = (float)(n / (double)p.N);
        const double lp = pf > 0.f ? log((double)pf) : pf == 0.f ? -CUDART_INF : CUDART_NAN;
        const double c = 1.4426950408889634074 * (lp - 0.5 * (((red[0] + red[1]) + red[2]) + red[3]));
        p.c2[k] = (float)c;
        p.c2d[k] = c;
    }
}

// ------------------------------------------------------------------------------------------------------------------
// A fit whose points fit into the shared memory of one cluster of 16 CTAs, and whose iterations are launches and trips to memory otherwise: one launch for
// all of them.  A CTA keeps its points; the parameters are in every CTA.  Per iteration: log-sum-exp with the responsibilities into shared memory (a point per
// 2^lgG lanes, four components each), statistics (a thread per tile of four components x four dimensions, FT / T replicas of them), both about the mean of the means, as
// DK_FUSED; the replicas' sums meet in float64, component k's of all CTAs in CTA k % 16, which updates it and writes its constants to all.  Two
// cluster barriers.
// Bound by the latency of that chain: 10K x 16, K = 8 (cycles of an iteration, about): centre 1300, log-sum-exp 5400, statistics 3000, replicas 2000, sums of all CTAs 2000,
// update 3300, barriers 1500.  Whole call, 10 iterations: 209 us with the launches, 153 now.
// Sums of many terms are taken in parts, at 1 % of the time: the CTAs' rows are many and the lanes of a point few, and errors of one sum after the other grow with the
// number of its terms (variances of 3000 x 60, K = 10 after an iteration 2.2e-7, in parts 8.3e-8, with the launches 8.3e-8).
constexpr double FIT_MOST = 6.5e6;
constexpr int FIT_SMEM = 220 * 1024;
constexpr int ST_NONE_NEW = 1 << 30;          // (a status that was there before)
constexpr int FT = 512, FC = 16, FIT_VALUES = 36, FIT_STRIDE = FT + 1;

struct FitArgs {
    const float* X;
    int64_t n;
    int D, K, P;             // points per CTA
    int D4, ld, ldr, kr, lgG, T, R, lgP, xvec;            // (2^lgP lanes share the replicas of an output)
    unsigned inv;            // tile * inv >> 16 = tile / D4
    float *pi, *mu, *var;
    float var_floor;
    int isotropic;
    double tol;
    double* ll;              // [slots] iteration i at i % slots
    int slots, first, end;   // iterations
    int *counts, *stop_at, *status;
};

__device__ __forceinline__ uint32_t fit_remote(const void* p, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ double fit_load(uint32_t a) { double v; asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ void fit_store(uint32_t a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void fit_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double fit_warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(FT, 1) direct_fit_kernel(const FitArgs p) {
    extern __shared__ __align__(16) float sm[];
    __shared__ double red_s[FT / 32], llr_s[FC];
    __shared__ __align__(16) float gs[128];
    __shared__ float pi_s[4];
    __shared__ int cnt_s[2], bad_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int D = p.D, K = p.K, D4 = p.D4, ld = p.ld, ldr = p.ldr, kr = p.kr, P = p.P, KD = K * D, W = 2 * D + 1;
    const int own = rank < K ? (K - rank + FC - 1) / FC : 0;             // this CTA's components: rank, rank + 16, ..
    double* const part = reinterpret_cast<double*>(sm);                  // [K + 2 K D + 1] N_k, sums, log-likelihood of this CTA's points
    double* const tmp = part + K + 2 * KD + 1;                           // [16][own][W] of all CTAs
    float* const sw = reinterpret_cast<float*>(tmp + FC * ((K + FC - 1) / FC) * W + (K + 1) % 2);         // [kr][ld] sqrt(w2)
    float* const ms = sw + kr * ld;                                      // (g - mu) sqrt(w2)
    float* const mean = ms + kr * ld;
    float* const cvs = mean + kr * ld;                                   // [kr]
    float* const vars = cvs + kr;                                        // [own][D]
    float* const xs = vars + ((K + FC - 1) / FC * D + 3) / 4 * 4;        // [P][ld]
    float* const rs = xs + P * ld;                                       // [P][ldr]
    const int64_t row0 = (int64_t)rank * P;
    const int mine = (int)(p.n - row0 < 0 ? 0 : p.n - row0 < P ? p.n - row0 : P);
    if (rank == 0 && tid < 2) p.counts[tid] = 0;
    if (tid == 0) bad_s = 0;
    __syncthreads();
    // ---- points and parameters
    for (int e = tid; e < P * D4; e += FT) {
        const int r = e / D4, c = 4 * (e - r * D4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < mine) {
            const float* src = p.X + (row0 + r) * D + c;
            if (p.xvec) v = __ldcg(reinterpret_cast<const float4*>(src));
            else {
                v.x = __ldcg(src);
                if (c + 1 < D) v.y = __ldcg(src + 1);
                if (c + 2 < D) v.z = __ldcg(src + 2);
                if (c + 3 < D) v.w = __ldcg(src + 3);
            }
        }
        *reinterpret_cast<float4*>(xs + r * ld + c) = v;
    }
    int bad = *p.status != 0 ? ST_NONE_NEW : 0;
    for (int k = warp; k < kr; k += FT / 32)
      for (int d = lane; d < 4 * D4; d += 32) {
        float w = 0.f, m = 0.f;
        if (k < K && d < D) {
            const float v = __ldcg(p.var + k * D + d);
            m = __ldcg(p.mu + k * D + d);
            if (!(v > 0.f) || !isfinite(v)) bad |= ST_BAD_VAR;
            if (!isfinite(m)) bad |= ST_NONFINITE;
            w = sqrtf((float)(0.72134752044448170368 / (double)v));
            if (k % FC == rank) vars[k / FC * D + d] = v;
        }
        sw[k * ld + d] = w;
        mean[k * ld + d] = m;
        ms[k * ld + d] = 0.f;
    }
    for (int k = warp; k < kr; k += FT / 32) {
        double lg = 0.0;
        if (k < K)
            for (int d = lane; d < D; d += 32) lg += log(6.283185307179586476925286766559 * (double)__ldcg(p.var + k * D + d));
        lg = fit_warp_sum(lg);
        if (lane == 0) {
            float c = -CUDART_INF_F;
            if (k < K) {
                const float w = __ldcg(p.pi + k);
                if (!(w >= 0.f) || !isfinite(w)) bad |= ST_BAD_PI;
                c = (float)(1.4426950408889634074 * ((w > 0.f ? log((double)w) : -CUDART_INF) - 0.5 * lg));
                if (k % FC == rank) pi_s[k / FC] = w;
            }
            cvs[k] = c;
        }
    }
    const int lgG = p.lgG, G = 1 << lgG, gq = lane & (G - 1);
    const int rep = tid / p.T, tt = tid - rep * p.T, dt = tt % D4, kt = tt / D4;
    double prev = p.first > 0 ? __ldcg(p.ll + (p.first - 1) % p.slots) : 0.0;
    const double rk = 1.0 / (double)K;
    bool updated = false, stop = false;
    int it = p.first;
    for (; it < p.end; ++it) {
        __syncthreads();
        if (tid < 2) cnt_s[tid] = 0;
        if (tid < 128) {
            double a = 0.0;
            if (tid < D)
#pragma unroll 8
                for (int k = 0; k < K; ++k) a += (double)mean[k * ld + tid];
            const float c = (float)(a * rk);
            gs[tid] = tid < D && isfinite(c) ? c : 0.f;
        }
        __syncthreads();
        for (int k = warp; k < K; k += FT / 32)
            for (int d = lane; d < D; d += 32) {
                const float m = mean[k * ld + d], w = sw[k * ld + d];
                if (!isfinite(m)) bad |= ST_NONFINITE;
                if (!(w > 0.f) || !isfinite(w)) bad |= ST_BAD_VAR;
                ms[k * ld + d] = (gs[d] - m) * w;
            }
        if (tid < K && isnan(cvs[tid])) bad |= ST_BAD_PI;
        __syncthreads();
        // ---- log-sum-exp, responsibilities
        double ll = 0.0;
        float cv[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) cv[b] = cvs[gq + G * b];
        auto points = [&](auto pts) {
            constexpr int PT = decltype(pts)::value;
            for (int base = warp * 32; base < P << lgG; base += PT * FT) {
                const float* xr[PT];
                u64 q[PT][4];
#pragma unroll
                for (int j = 0; j < PT; ++j) {
                    xr[j] = xs + min((base + j * FT + lane) >> lgG, P - 1) * ld;
#pragma unroll
                    for (int b = 0; b < 4; ++b) q[j][b] = 0ull;
                }
                // (eight or sixteen dimensions at a time, which are added to the others then: half the error of one sum of all)
                auto dims = [&](int d4, auto steps) {
                    constexpr int ST = decltype(steps)::value;
                    ulonglong2 x[PT][ST];
#pragma unroll
                    for (int s = 0; s < ST; ++s) {
                        const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gs + 4 * (d4 + s));
#pragma unroll
                        for (int j = 0; j < PT; ++j) {
                            x[j][s] = *reinterpret_cast<const ulonglong2*>(xr[j] + 4 * (d4 + s));
                            x[j][s].x = fma2(g.x, 0xBF800000BF800000ull, x[j][s].x);
                            x[j][s].y = fma2(g.y, 0xBF800000BF800000ull, x[j][s].y);
                        }
                    }
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        u64 f[PT];
#pragma unroll
                        for (int s = 0; s < ST; ++s) {
                            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(sw + (gq + G * b) * ld + 4 * (d4 + s));
                            const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(ms + (gq + G * b) * ld + 4 * (d4 + s));
#pragma unroll
                            for (int j = 0; j < PT; ++j) {
                                const u64 t0 = fma2(x[j][s].x, w.x, m.x), t1 = fma2(x[j][s].y, w.y, m.y);
                                f[j] = s == 0 ? mul2(t0, t0) : fma2(t0, t0, f[j]);
                                f[j] = fma2(t1, t1, f[j]);
                            }
                        }
#pragma unroll
                        for (int j = 0; j < PT; ++j) q[j][b] = add2(q[j][b], f[j]);
                    }
                };
                constexpr int MOST = PT == 3 ? 2 : 4;        // (of three points the coordinates do not fit the registers)
                int d4 = 0;
#pragma unroll 1
                for (; d4 + MOST <= D4; d4 += MOST) dims(d4, std::integral_constant<int, MOST>{});
                if (MOST > 2 && d4 + 2 <= D4) {
                    dims(d4, std::integral_constant<int, 2>{});
                    d4 += 2;
                }
                if (d4 < D4) dims(d4, std::integral_constant<int, 1>{});
                float l[PT][4], m[PT], a[PT];
#pragma unroll
                for (int j = 0; j < PT; ++j) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) l[j][b] = cv[b] - (lo2(q[j][b]) + hi2(q[j][b]));
                    m[j] = fmaxf(fmaxf(l[j][0], l[j][1]), fmaxf(l[j][2], l[j][3]));
                }
                for (int o = 1; o < G; o <<= 1)
#pragma unroll
                    for (int j = 0; j < PT; ++j) m[j] = fmaxf(m[j], __shfl_xor_sync(0xffffffffu, m[j], o));
#pragma unroll
                for (int j = 0; j < PT; ++j) {
                    const float ref = m[j] == -CUDART_INF_F ? 0.f : m[j];
                    a[j] = 0.f;
#pragma unroll
                    for (int b = 0; b < 4; ++b) { l[j][b] = dk_ex2(l[j][b] - ref); a[j] += l[j][b]; }
                }
                for (int o = 1; o < G; o <<= 1)
#pragma unroll
                    for (int j = 0; j < PT; ++j) a[j] += __shfl_xor_sync(0xffffffffu, a[j], o);
#pragma unroll
                for (int j = 0; j < PT; ++j) {
                    const int pt = (base + j * FT + lane) >> lgG;
                    const bool in = pt < mine;
                    if (in && gq == 0) ll += (double)m[j] + (double)log2f(a[j]);
                    const float f = in ? 1.0f / a[j] : 0.f;
                    if (pt < P) {
#pragma unroll
                        for (int b = 0; b < 4; ++b)
                            if (gq + G * b < ldr) rs[pt * ldr + gq + G * b] = in ? l[j][b] * f : 0.f;
                    }
                }
            }
        };
        // (as many points per lane at once as there are rounds, up to three: the rounds' latencies overlap)
        const int rounds = ((P << lgG) + FT - 1) / FT;
        if (rounds == 1) points(std::integral_constant<int, 1>{});
        else if (rounds == 2) points(std::integral_constant<int, 2>{});
        else points(std::integral_constant<int, 3>{});
        ll = fit_warp_sum(ll);
        if (lane == 0) red_s[warp] = ll;
        __syncthreads();
        // ---- statistics
        u64 a1[4][2], a2[4][2];
        float nacc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 4; ++c) a1[c][0] = a1[c][1] = a2[c][0] = a2[c][1] = 0ull;
        if (rep < p.R) {
            const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gs + 4 * dt);
            auto row = [&](int r, u64 (&f1)[4][2], u64 (&f2)[4][2], float (&fn)[4]) {
                ulonglong2 x = *reinterpret_cast<const ulonglong2*>(xs + r * ld + 4 * dt);
                x.x = fma2(g.x, 0xBF800000BF800000ull, x.x);
                x.y = fma2(g.y, 0xBF800000BF800000ull, x.y);
                const u64 y0 = mul2(x.x, x.x), y1 = mul2(x.y, x.y);
                const float4 w = *reinterpret_cast<const float4*>(rs + r * ldr + 4 * kt);
                const float rr[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const u64 rd = dup2(rr[c]);
                    fn[c] += rr[c];
                    f1[c][0] = fma2(rd, x.x, f1[c][0]);
                    f1[c][1] = fma2(rd, x.y, f1[c][1]);
                    f2[c][0] = fma2(rd, y0, f2[c][0]);
                    f2[c][1] = fma2(rd, y1, f2[c][1]);
                }
            };
            // (four rows at a time, the last ones too, which are added to the others then: half the error of one sum of all)
#pragma unroll 1
            for (int r = rep; r < mine; r += 4 * p.R) {
                u64 f1[4][2], f2[4][2];
                float fn[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int c = 0; c < 4; ++c) f1[c][0] = f1[c][1] = f2[c][0] = f2[c][1] = 0ull;
                if (r + 3 * p.R < mine) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) row(r + u * p.R, f1, f2, fn);
                } else {
#pragma unroll 1
                    for (int t = r; t < mine; t += p.R) row(t, f1, f2, fn);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    nacc[c] += fn[c];
#pragma unroll
                    for (int h = 0; h < 2; ++h) { a1[c][h] = add2(a1[c][h], f1[c][h]); a2[c][h] = add2(a2[c][h], f2[c][h]); }
                }
            }
        }
        __syncthreads();                                     // (the responsibilities have been read)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float* const o = rs + 8 * c * FIT_STRIDE + tid;
            o[0] = lo2(a1[c][0]); o[FIT_STRIDE] = hi2(a1[c][0]); o[2 * FIT_STRIDE] = lo2(a1[c][1]); o[3 * FIT_STRIDE] = hi2(a1[c][1]);
            o[4 * FIT_STRIDE] = lo2(a2[c][0]); o[5 * FIT_STRIDE] = hi2(a2[c][0]); o[6 * FIT_STRIDE] = lo2(a2[c][1]); o[7 * FIT_STRIDE] = hi2(a2[c][1]);
            rs[(32 + c) * FIT_STRIDE + tid] = nacc[c];
        }
        __syncthreads();
        // (a warp has a value of all tiles; neighbouring lanes share a tile's replicas)
        for (int i = warp; i < FIT_VALUES; i += FT / 32)
            for (int t0 = 0; t0 < p.T; t0 += 32 >> p.lgP) {
                const int tile = t0 + (lane >> p.lgP), q = lane & ((1 << p.lgP) - 1);
                double a[2] = {0.0, 0.0};
                if (tile < p.T) {
                    const float* const v = rs + i * FIT_STRIDE + tile;
#pragma unroll 4
                    for (int r = q; r < p.R; r += 2 << p.lgP) {
                        a[0] += (double)v[r * p.T];
                        if (r + (1 << p.lgP) < p.R) a[1] += (double)v[(r + (1 << p.lgP)) * p.T];
                    }
                }
                double t = a[0] + a[1];
                for (int x = 1; x < 1 << p.lgP; x <<= 1) t += __shfl_xor_sync(0xffffffffu, t, x);
                const int row = (int)(((unsigned)tile * p.inv) >> 16), col = tile - row * D4, k = 4 * row + (i < 32 ? i >> 3 : i - 32), d = 4 * col + (i & 3);
                if (tile < p.T && q == 0 && k < K && (i < 32 ? d < D : col == 0)) part[i >= 32 ? k : K + (i & 4 ? KD : 0) + k * D + d] = t;
            }
        if (tid == 0) {
            double a = 0.0;
            for (int w = 0; w < FT / 32; ++w) a += red_s[w];
            part[K + 2 * KD] = a * 0.69314718055994530942;
        }
        if (bad) atomicOr(&bad_s, bad);
        __syncthreads();
        bad = bad_s;                                         // (the same in every CTA)
        fit_barrier();
        // ---- all CTAs' sums of this CTA's components; everyone needs to know what becomes of the iteration
        if (tid < FC) llr_s[tid] = fit_load(fit_remote(part + K + 2 * KD, tid));
        static_assert(FT / 32 == FC, "a warp per CTA");
        for (int kc = 0; kc < own; ++kc) {
            const int k = rank + FC * kc;
            for (int out = lane; out < W; out += 32)
                tmp[(warp * own + kc) * W + out] = fit_load(fit_remote(part + (out == 0 ? k : out <= D ? K + k * D + out - 1 : K + KD + k * D + out - 1 - D), warp));
        }
        __syncthreads();
        for (int o = tid; o < own * W; o += FT) {
            double a = 0.0;
#pragma unroll
            for (int src = 0; src < FC; ++src) a += tmp[src * own * W + o];
            tmp[o] = a;
        }
        ll = 0.0;
#pragma unroll
        for (int src = 0; src < FC; ++src) ll += llr_s[src];
        __syncthreads();
        const bool good = bad == 0 && isfinite(ll);          // a step that failed leaves the parameters as they are
        stop = !good || (p.tol > 0.0 && it > 0 && fabs(ll - prev) <= p.tol * fabs(ll));
        prev = ll;
        if (rank == 0 && tid == 0) p.ll[it % p.slots] = ll;
        if (good) {
            updated = true;
            for (int kc = warp; kc < own; kc += FT / 32) {
                const int k = rank + FC * kc;
                const double* const t = tmp + kc * W;
                const double n = t[0];
                const bool empty = n < 1e-12;                // an empty component keeps mu and var
                const double rn = 1.0 / n;
                const float pf = (float)(n / (double)p.n);   // pi_k = N_k / N
                const double lp = pf > 0.f ? log((double)pf) : pf == 0.f ? -CUDART_INF : CUDART_NAN;
                double vd[4], vsum = 0.0, lg = 0.0;
                int floored = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int d = lane + 32 * i;
                    vd[i] = 0.0;
                    if (d >= D || empty) continue;
                    const double g = (double)gs[d], s1 = t[1 + d] + g * n, s2 = t[1 + D + d] + 2.0 * g * t[1 + d] + g * g * n, m = s1 * rn;      // Eq. 2
                    vd[i] = s2 * rn - m * m;                 // Eq. 3 per dimension, new mean
                    vsum += vd[i];
                    for (int c = 0; c < FC; ++c) fit_store(fit_remote(mean + k * ld + d, c), (float)m);
                }
                const double fl = (double)p.var_floor;
                if (p.isotropic) {                           // one variance: the mean over the dimensions
                    vsum = fit_warp_sum(vsum) / (double)D;
                    if (!empty && !(vsum > fl)) { vsum = fl; if (lane == 0) floored = D; }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int d = lane + 32 * i;
                    if (d >= D) continue;
                    if (!empty) {
                        double v = p.isotropic ? vsum : vd[i];
                        if (!p.isotropic && !(v > fl)) { v = fl; ++floored; }
                        vars[kc * D + d] = (float)v;
                    }
                    const float vf = vars[kc * D + d];
                    lg += log(6.283185307179586476925286766559 * (double)vf);
                    const float w = sqrtf((float)(0.72134752044448170368 / (double)vf));
                    for (int c = 0; c < FC; ++c) fit_store(fit_remote(sw + k * ld + d, c), w);
                }
                lg = fit_warp_sum(lg);
                floored = __reduce_add_sync(0xffffffffu, floored);
                if (lane < FC) fit_store(fit_remote(cvs + k, lane), (float)(1.4426950408889634074 * (lp - 0.5 * lg)));
                if (lane == 0) {
                    pi_s[kc] = pf;
                    if (floored) atomicAdd(&cnt_s[0], floored);
                    if (empty) atomicAdd(&cnt_s[1], 1);
                }
            }
        }
        __syncthreads();
        fit_barrier();
        if (stop) break;
    }
    if (updated) {
        __syncthreads();
        for (int e = tid; e < own * D; e += FT) {
            const int kc = e / D, d = e - kc * D, k = rank + FC * kc;
            p.mu[(size_t)k * D + d] = mean[k * ld + d];
            p.var[(size_t)k * D + d] = vars[e];
        }
        if (tid < own) p.pi[rank + FC * tid] = pi_s[tid];
        if (tid < 2 && cnt_s[tid]) atomicAdd(p.counts + tid, cnt_s[tid]);
    }
    if (rank == 0 && tid == 0) {
        *p.stop_at = stop ? it : 0x7f7f7f7f;
        if (bad & ~ST_NONE_NEW) atomicOr(p.status, bad & ~ST_NONE_NEW);
    }
}

// ------------------------------------------------------------------------------------------------------------------
struct DirectPlan {
    DirectArgs a;
    int PT, TK;
    int64_t tiles;
    size_t smem;
    int per_sm;
};

constexpr int SMS = 148;

// Shape of the tiles for n points.
DirectPlan direct_plan(int mode, const float* X, int64_t n, int D, int K) {
    DirectPlan pl{};
    DirectArgs& a = pl.a;
    a.X = X; a.n = n; a.D = D; a.K = K;
    const int kb = K < 64 ? K : 64, cblocks = mode == DK_STATS ? (K + 63) / 64 : 1;
    a.D4 = (D + 3) / 4;
    // rows of x and of the parameters: an odd multiple of the 16 S bytes that the S lanes of a point read (no bank conflicts)
    auto set_ld = [&]() { a.ld = 4 * (((a.D4 + (1 << a.lgS) - 1) >> a.lgS) | 1) << a.lgS; };
    set_ld();
    while ((4 << a.lgG) < kb) ++a.lgG;
    a.kr = 4 << a.lgG;
    while ((1 << a.lgX) < a.D4) ++a.lgX;
    a.xvec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    // four components per tile of the statistics where eight would be padding (and the tiles fit the threads)
    pl.TK = 8;
    if (((kb - 1) & 7) < 4 && (kb + 3) / 4 * a.D4 <= NT) pl.TK = 4;
    const int kp = (kb + pl.TK - 1) / pl.TK * pl.TK;
    a.ldr = 4 * ((kp / 4) | 1);
    a.T = kp / pl.TK * a.D4;
    a.R = NT / a.T;
    // points per tile: four per lane, fewer where the tile would not leave room for a second CTA on the SM, or where there would
    // not be a tile for every SM; the lanes then share the dimensions as long as there are eight per lane
    pl.PT = (mode == DK_LSE || D > 32) ? 4 : 2;          // (at four, the statistics' registers spill, once per tile)
    a.NS = 1;
    auto tp = [&]() { return (int64_t)a.NS * pl.PT * (NT >> (a.lgG + a.lgS)); };
    const int nblk = mode == DK_LSE ? (K + 63) / 64 : 1, row_extra = mode == DK_FUSED ? a.ldr : mode == DK_STATS ? a.ldr + 1 : nblk > 1 ? 2 : 0;
    auto bytes = [&]() { return (2 * a.kr * a.ld + tp() * (a.ld + row_extra)) * 4; };
    while (bytes() > 110592 || (n + tp() - 1) / tp() * cblocks < SMS) {
        if (a.lgG + a.lgS < 5 && a.D4 >= (4 << a.lgS)) { ++a.lgS; set_ld(); }
        else if (pl.PT > 1) pl.PT >>= 1;
        else break;
    }
    // few dimensions: a tile's barriers (and, with several blocks of components, their parameters) cost more than its arithmetic, so a
    // tile takes more points as long as there are tiles for all SMs
    while (a.NS < 16 && a.NS * a.D4 < 32 && (pl.PT < 4 || mode == DK_LSE)) {
        a.NS *= 2;
        if (bytes() > 110592 || (n + tp() - 1) / tp() * cblocks < 2 * SMS) { a.NS /= 2; break; }
    }
    pl.tiles = (n + tp() - 1) / tp();
    size_t fl = (size_t)2 * a.kr * a.ld + (size_t)tp() * (a.ld + row_extra);
    if (mode != DK_LSE && a.R > 1 && fl < (size_t)8 * pl.TK * (NT + a.T)) fl = (size_t)8 * pl.TK * (NT + a.T);
    pl.smem = fl * 4;
    pl.per_sm = pl.smem + 6144 <= 233472 / 2 ? 2 : 1;
    return pl;
}

template <typename Args>
cudaError_t launch_chained(cudaStream_t s, dim3 grid, int threads, size_t smem, void (*kernel)(Args), const Args& a) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}
constexpr int MOST_SMEM = 114688;          // (no shape asks for more than 110592 bytes, see direct_plan)
template <int MODE, int PT, int TK>
cudaError_t direct_launch(cudaStream_t s, dim3 grid, const DirectPlan& pl) {
    if (pl.smem > 40960) {
        // (the same limit from every call: it belongs to the kernel, which contexts on other threads launch for other shapes)
        cudaError_t e = cudaFuncSetAttribute(direct_kernel<MODE, PT, TK>, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST_SMEM);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(s, grid, NT, pl.smem, direct_kernel<MODE, PT, TK>, pl.a);
}
template <int MODE>
cudaError_t direct_launch(cudaStream_t s, dim3 grid, const DirectPlan& pl) {
    const bool t8 = MODE != DK_LSE && pl.TK == 8;
    switch (pl.PT) {
        case 1: return t8 ? direct_launch<MODE, 1, 8>(s, grid, pl) : direct_launch<MODE, 1, 4>(s, grid, pl);
        case 2: return t8 ? direct_launch<MODE, 2, 8>(s, grid, pl) : direct_launch<MODE, 2, 4>(s, grid, pl);
        default: return t8 ? direct_launch<MODE, 4, 8>(s, grid, pl) : direct_launch<MODE, 4, 4>(s, grid, pl);
    }
}

}  // namespace

int lse_direct_parts(int64_t n, int D, int K) {
    const DirectPlan pl = direct_plan(DK_LSE, nullptr, n, D, K);
    return (int)(pl.tiles < SMS * pl.per_sm ? pl.tiles : SMS * pl.per_sm);
}

cudaError_t launch_lse_direct(cudaStream_t s, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                              const double* c2d, const float* g, double* logZ2, double* llpart) {
    DirectPlan pl = direct_plan(DK_LSE, X, n, D, K);
    pl.a.mu = mu; pl.a.w2 = w2; pl.a.c2d = c2d; pl.a.g = g; pl.a.logZ2 = logZ2; pl.a.llpart = llpart; pl.a.ll_first = 1;
    return direct_launch<DK_LSE>(s, dim3((unsigned)lse_direct_parts(n, D, K)), pl);
}

cudaError_t launch_mstep_direct(cudaStream_t s, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                                const double* c2d, const float* g, const double* logZ2, float* partials, int splits) {
    DirectPlan pl = direct_plan(DK_STATS, X, n, D, K);
    pl.a.mu = mu; pl.a.w2 = w2; pl.a.c2d = c2d; pl.a.g = g; pl.a.logZ2 = const_cast<double*>(logZ2); pl.a.partials = partials;
    return direct_launch<DK_STATS>(s, dim3((unsigned)splits, (unsigned)((K + 63) / 64)), pl);
}

cudaError_t launch_reduce_direct(cudaStream_t s, int D, int K, int splits, const float* partials, const float* g, double* Nk,
                                 double* S1, double* S2, bool accumulate) {
    ReduceArgs r{};
    r.D = D; r.K = K; r.splits = splits; r.partials = partials; r.g = g; r.Nk = Nk; r.S1 = S1; r.S2 = S2; r.accumulate = accumulate ? 1 : 0;
    return launch_chained(s, dim3((unsigned)K), 1024, 0, direct_reduce_kernel, r);
}

// Where one launch is the faster way: 16 SMs take about as long for a point and component as for 16 dimensions more, two launches per iteration 14 to 20 us
// (whole fits of five iterations, us, launches / one launch: 5K x 64, K = 16 204 / 159, 20K x 16, K = 8 143 / 125, 5K x 16, K = 32 154 / 133, 10K x 32, K = 8
// 150 / 120, 2K x 4, K = 3 147 / 89; beyond the line 20K x 16, K = 16 153 / 170, 100K x 4, K = 4 150 / 134).
static bool fit_plan(const float* X, int64_t n, int D, int K, FitArgs* out, size_t* smem) {
    if (D > 128 || K > 64 || K * D > 1024 || (double)n * K * (D + 16) > FIT_MOST) return false;
    FitArgs a{};
    a.X = X; a.n = n; a.D = D; a.K = K;
    a.P = (int)((n + FC - 1) / FC);
    a.D4 = (D + 3) / 4;
    a.ld = 4 * (a.D4 | 1);
    while ((4 << a.lgG) < K) ++a.lgG;
    a.kr = 4 << a.lgG;
    const int k4 = (K + 3) / 4;
    a.ldr = 4 * (k4 | 1);
    a.T = k4 * a.D4;
    a.R = FT / a.T;
    while ((a.T << (a.lgP + 1)) <= 32) ++a.lgP;
    a.inv = (65536u + a.D4 - 1) / a.D4;                      // (exact below 65536 / D4: at most 256 tiles of 32 columns)
    a.xvec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    const size_t rs = (size_t)a.P * a.ldr, sums = (size_t)FIT_VALUES * FIT_STRIDE;
    const int most = (K + FC - 1) / FC, W = 2 * D + 1;
    size_t bytes = 8 * (size_t)(K + 2 * K * D + 1 + FC * most * W + (K + 1) % 2);
    bytes += 4 * ((size_t)3 * a.kr * a.ld + a.kr + (most * D + 3) / 4 * 4 + (size_t)a.P * a.ld + (rs > sums ? rs : sums));
    if (bytes > FIT_SMEM) return false;
    *out = a;
    *smem = bytes;
    return true;
}
bool fit_direct_supports(const float* X, int64_t n, int D, int K) {
    FitArgs a;
    size_t smem;
    return fit_plan(X, n, D, K, &a, &smem);
}
cudaError_t launch_fit_direct(cudaStream_t s, const float* X, int64_t n, int D, int K, const DirectFit& f, double* ll, int slots, int end, int* status) {
    FitArgs a;
    size_t smem;
    if (!fit_plan(X, n, D, K, &a, &smem)) return cudaErrorInvalidValue;
    a.pi = f.pi; a.mu = f.mu; a.var = f.var; a.var_floor = f.var_floor; a.isotropic = f.isotropic ? 1 : 0; a.tol = f.tol;
    a.ll = ll; a.slots = slots; a.first = f.iter; a.end = end; a.counts = f.counts; a.stop_at = f.stop_at; a.status = status;
    // (the same limits from every call: they belong to the kernel)
    cudaError_t e = cudaFuncSetAttribute(direct_fit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FIT_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(direct_fit_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(FC); cfg.blockDim = dim3(FT); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = FC; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    cfg.attrs = &at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, direct_fit_kernel, a);
}

bool fused_direct_supports(int D, int K) { return D <= 128 && K <= 64; }

cudaError_t launch_fused_direct(cudaStream_t s, const float* X, int64_t n, int D, int K, const float* mu, float* w2, float* c2,
                                double* c2d, float* g, float* partials, double* llpart, double* Nk, double* S1, double* S2,
                                bool accumulate, double* ll, int* status, const DirectFit* fit, int64_t* launches) {
    // an fp32 sum takes at most 4096 points: beyond that (per replica and CTA) the points go in several launches, whose statistics
    // are added in float64
    DirectPlan pl = direct_plan(DK_FUSED, X, n, D, K);
    const int64_t ctas = pl.tiles < (int64_t)SMS * pl.per_sm ? pl.tiles : (int64_t)SMS * pl.per_sm;
    const int64_t piece = ctas * pl.a.R * 4096;
    for (int64_t off = 0; off < n; off += piece) {
        const int64_t cnt = n - off < piece ? n - off : piece;
        const bool last = off + cnt == n;
        DirectArgs& a = pl.a;
        a.X = X + off * D; a.n = cnt;
        a.xvec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(a.X) & 15) == 0);
        a.mu = mu; a.w2 = w2; a.c2d = c2d; a.g_out = g; a.llpart = llpart; a.ll_first = off == 0 ? 1 : 0; a.partials = partials;
        a.status = status;
        if (fit) { a.counts = fit->counts; a.stop_at = fit->stop_at; a.iter = fit->iter; }
        const int64_t tp = (int64_t)a.NS * pl.PT * (NT >> (a.lgG + a.lgS)), tiles = (cnt + tp - 1) / tp;
        const int grid = (int)(tiles < ctas ? tiles : ctas);
        cudaError_t e = direct_launch<DK_FUSED>(s, dim3((unsigned)grid), pl);
        if (e != cudaSuccess) return e;
        ReduceArgs r{};
        r.D = D; r.K = K; r.splits = grid; r.partials = partials; r.g = g; r.Nk = Nk; r.S1 = S1; r.S2 = S2;
        r.accumulate = (accumulate || off > 0) ? 1 : 0;
        if (last) { r.llpart = llpart; r.n_ll = (int)ctas; r.ll = ll; r.ll_accumulate = accumulate ? 1 : 0; }
        if (fit) {
            r.stop_at = fit->stop_at; r.iter = fit->iter;
            if (last) {
                r.pi = fit->pi; r.mu = fit->mu; r.var = fit->var; r.var_floor = fit->var_floor; r.isotropic = fit->isotropic ? 1 : 0; r.N = n;
                r.counts = fit->counts; r.status = status; r.w2 = w2; r.c2 = c2; r.c2d = c2d; r.ll_prev = fit->ll_prev; r.tol = fit->tol;
            }
        }
        e = launch_chained(s, dim3((unsigned)K), 1024, 0, direct_reduce_kernel, r);
        if (e != cudaSuccess) return e;
        *launches += 2;
    }
    return cudaSuccess;
}

}  // namespace fg
