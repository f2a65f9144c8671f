// The screening path for D <= 128 (sm_100a, tcgen05 + TMEM): few (point, component) pairs of a mixture matter.
//
// Where posteriors are sparse - a handful of components within 2^-40 of a point's best - only those pairs need their exact
// densities and statistics.  ONE sweep of the tensor cores over a single fp16 product per contraction (a sixth of the work of
// the kernels that form every responsibility from split operands) tells which they are, with rigorous error bounds:
//
//   screen_sweep_kernel   TMEM lanes = points.  A CTA holds the fp16 rows of 256 points in tensor memory and streams the
//                         components' coefficients past them, 128 at a time; a softmax thread owns one point, keeps the largest
//                         lower bound seen so far and the components whose upper bound reaches it (less the margin), drops
//                         those that the final bound rules out, and writes the rest as a list.
//   screen_eval_kernel    the listed pairs in fp32 direct differences: log-sum-exp, responsibilities, or the arg-max.
//   screen_scan/fill/stats/reduce   the kept pairs sorted by component (stable, no atomics on the output), streamed as rows of
//                         X against the component's mean in registers, fp32 within 64 pairs, float64 beyond.
//
// Every value that reaches a result comes from exact fp32 evaluations; a term below 2^-40 of a point's total is dropped.  Data
// whose posteriors are broad is noticed ahead of the sweep, from a sample of the rows (screen_probe), or at the latest behind the sweep of a
// piece (SC_DENSE): the kernels that follow return at once and the caller runs the dense kernels instead.
#include "em_screen.cuh"
#include "internal.cuh"

#define TC_WAIT_LIMIT_NS 2000000000ull
#include "tc_prims.cuh"

namespace fg {

namespace {

// ------------------------------------------------------------------------------------------------------------------
// Parameter preparation
//
// Points and means enter as u = s_d (x - g_d), nu = s_d (mu - g_d): g the mixture's mean, s_d a power of two that brings the
// dimension to size 1.  With b = w2 / s^2 (w2 = log2 e / (2 var)):  log2 z = c + sum_d (2 b nu) u + (-b) u^2,
// c = log2 pi + ... - sum_d b nu^2.  The coefficients are rounded to fp16 as they are; c is split into three fp16 values (of 256,
// 1 and 1) and added by the tensor cores too, so that an accumulator IS the approximate log2 z: a table of scales and constants
// read by every softmax thread cost more shared-memory bandwidth than the products.
//
// Error of the approximate log2 z of ANY point: u and the coefficients are rounded to 2^-11 (or to 2^-25, the spacing of
// subnormals), the square of the rounded u once more (3 x 2^-11 in all), and the products are added into an fp32 accumulator
// that loses less than 2^-18 of the terms' sizes:  2^-10 sum_d 2 b |nu u| + 2^-9 sum_d b u^2 <= 2^-10 (sum_d b nu^2 + 3 max_d b |u|^2).
// So it is below alpha + beta |u|^2 with
//   alpha = eps sum_d b nu^2 + 2^-24 sum_d (2 b |nu| + b) + 2^-25 D / 2 + 2^-18 |c| + 0.02
//   beta  = 3 eps max_d b + 1.5 x 2^-25,        eps = 2^-10 (1 + 2^-6).
//
// A component that is much narrower than the data in some dimensions (a few points, one point) has a huge max_d b, and with it
// an allowance that rules nothing out (or coefficients beyond fp16).  Where the allowance of a typical point exceeds SCR_SHARP
// bits, b is CAPPED at a value that leaves about 16: c - sum_d min(b, cap) (u - nu)^2 is an upper bound of log2 z, which is what
// the screening needs, with a small allowance; only its lower bound is lost, so such components do not raise the threshold.
//
// k-means (unit): every component has the same weights, so sum_d b u^2 is the same for all of them and drops out of every comparison that
// the sweep makes: the contraction has the linear terms alone, half as long, and
//   alpha = eps sum_d b nu^2 + 2^-24 sum_d (2 b |nu| + b) + 2^-25 D / 2 + 2^-18 |c| + 0.02,   beta = eps max_d b + 1.5 x 2^-25.
// The weight is F = min(1, min_d s_d^2) instead of 1, a power of two: with it b <= 1, and data larger than size 1 are screened in units in
// which the allowances are small (with weight 1 data ten times as large have allowances a hundred times as large).  Smaller data keep
// weight 1, where the 0.02 of alpha is a squared distance like any other: it counts from where the two nearest centroids are about as close.
// (Clusters of vectors of unit norm are screened as others, 300K x 96, K = 1024 292 us against 285.  F > 1 would have to look at X as well:
// points far from centroids that are close to one another leave float32.)
constexpr float SCR_SHARP = 40.f;
constexpr float SCR_CAPPED = 1e30f;          // their sorting key
constexpr float SCR_NEVER = -1.5e7f;         // c of a position without a component
// (numax: largest |nu| of the component; 2 cap |nu| stays within fp16)
__device__ __forceinline__ double screen_cap(int D, double numax) { return fmin(fmin(16.0 / (3.0 * 9.765625e-04 * (double)D), 30000.0), 30000.0 / fmax(numax, 1e-30)); }

__global__ void __launch_bounds__(512) screen_dim_kernel(int D, int K, const float* __restrict__ pi, const float* __restrict__ mu,
                                                         const float* __restrict__ var, int unit, double* __restrict__ part,
                                                         float* __restrict__ sd, float* __restrict__ gd, int* __restrict__ ctl) {
    __shared__ double sum[4][512];
    __shared__ int last_s;
    const int tid = threadIdx.x, d = tid & 127, r = tid >> 7;
    double m0 = 0.0, m1 = 0.0, m2 = 0.0, v = 0.0;
    const int stride = gridDim.x * 4;
    for (int k0 = blockIdx.x * 4 + r; k0 < K; k0 += 4 * stride) {
        float p[4], m[4], w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u * stride;
            const bool in = k < K && d < D;
            p[u] = k < K ? (unit ? 1.f : __ldg(pi + k)) : 0.f;
            m[u] = in ? __ldg(mu + (size_t)k * D + d) : 0.f;
            w[u] = in && !unit ? __ldg(var + (size_t)k * D + d) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const double pd = (double)p[u], md = (double)m[u];
            m0 += pd;
            m1 += pd * md;
            m2 += pd * md * md;
            v += pd * (double)w[u];
        }
    }
    sum[0][tid] = m0; sum[1][tid] = m1; sum[2][tid] = m2; sum[3][tid] = v;
    __syncthreads();
    // (thread = quantity r of dimension d)
    part[(size_t)blockIdx.x * 512 + tid] = sum[r][d] + sum[r][128 + d] + sum[r][256 + d] + sum[r][384 + d];
    __threadfence();
    __syncthreads();
    if (tid == 0) last_s = atomicAdd(ctl + SC_TICKET_A, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last_s) return;
    // the last CTA to finish adds the partial sums in order
    __threadfence();
    double t = 0.0;
    for (int b0 = 0; b0 < (int)gridDim.x; b0 += 16) {
        double q[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) q[u] = b0 + u < (int)gridDim.x ? __ldcg(part + (size_t)(b0 + u) * 512 + tid) : 0.0;
#pragma unroll
        for (int u = 0; u < 16; ++u) t += q[u];
    }
    sum[r][d] = t;
    __syncthreads();
    if (r != 0) return;
    m0 = sum[0][d]; m1 = sum[1][d]; m2 = sum[2][d]; v = sum[3][d];
    float gf = m0 > 0.0 ? (float)(m1 / m0) : 0.f;
    if (!isfinite(gf) || d >= D) gf = 0.f;
    float s = 1.f;
    if (m0 > 0.0 && d < D) {
        const double g = (double)gf;
        const double ms = (m2 - 2.0 * g * m1 + g * g * m0 + v) / m0;
        if (ms > 0.0 && isfinite(ms)) s = (float)exp2(-fmin(fmax(rint(0.5 * log2(ms)), -60.0), 60.0));
    }
    sd[d] = s;
    gd[d] = gf;
    if (d == 0) {
        ctl[SC_MARKS] = 0;
        ctl[SC_OVF] = 0;
        ctl[SC_EXTRA] = 0;
        ctl[SC_TICKET_A] = 0;
        ctl[SC_PROBED] = 0;
        ctl[SC_DONE] = 0;
        ctl[SC_DENSE] = 0;
        ctl[SC_ACTIVE] = 0;
        ctl[SC_KEPT] = 0;
    }
}

// Whether the call has been left to the dense kernels, the same for all threads of the CTA: one of them reads the word.  For kernels in which a
// CTA may find that out while another one starts: read by every thread for itself, some warps would leave and the others go on without them.
__device__ __forceinline__ bool screen_off(const int* ctl) { return __syncthreads_or(threadIdx.x == 0 && __ldcg(ctl + SC_DENSE) != 0) != 0; }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// F of the unit mixture, the same in every lane.
__device__ __forceinline__ float screen_unit_weight(int D, const float* __restrict__ sd, int lane) {
    float f = 1.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (lane + 32 * i < D) { const float s = __ldg(sd + lane + 32 * i); f = fminf(f, s * s); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f = fminf(f, __shfl_xor_sync(0xffffffffu, f, o));
    return f;
}

// A warp per component: the FP32 kernels' derived parameters, the row's scale and constant, and the allowances above.
__global__ void __launch_bounds__(256) screen_comp_kernel(int D, int K, const float* __restrict__ pi, const float* __restrict__ mu,
                                                          const float* __restrict__ var, int unit, const float* __restrict__ sd,
                                                          const float* __restrict__ gd, float* __restrict__ w2, float* __restrict__ c2,
                                                          double* __restrict__ c2d, float4* __restrict__ prm, float* __restrict__ key,
                                                          int4* __restrict__ blk, unsigned* __restrict__ probe, double* __restrict__ ll, int* __restrict__ ctl,
                                                          int* __restrict__ status) {
    const int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x < SCR_MAX_K / 32) blk[threadIdx.x] = make_int4(0, 0, 0, 0);      // (largest allowances, see below)
    if (blockIdx.x == 0 && threadIdx.x < PR_GROUPS * (PR_ROWS + 1)) probe[threadIdx.x] = 0u;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < SCR_LL + K; i += gridDim.x * 256) ll[i] = 0.0;
    if (k >= K) return;
    double slog = 0.0, bv[4], nv[4];
    int bad = 0;
    const float F = unit ? screen_unit_weight(D, sd, lane) : 1.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int d = lane + 32 * i;
        bv[i] = nv[i] = 0.0;
        if (d >= D) continue;
        const float v = unit ? 1.f : __ldg(var + (size_t)k * D + d), m = __ldg(mu + (size_t)k * D + d);
        if (!(v > 0.f) || !isfinite(v)) bad |= ST_BAD_VAR;
        if (!isfinite(m)) bad |= ST_NONFINITE;
        const double w = unit ? (double)F : 0.72134752044448170368 / (double)v;
        if (!unit) slog += log(6.283185307179586476925286766559 * (double)v);
        w2[(size_t)k * D + d] = (float)w;
        const double s = (double)__ldg(sd + d);
        nv[i] = ((double)m - (double)__ldg(gd + d)) * s;
        bv[i] = w / (s * s);
    }
    slog = warp_sum(slog);
    bad = __reduce_or_sync(0xffffffffu, (unsigned)bad);
    const float p = unit ? 1.f : __ldg(pi + k);
    if (!(p >= 0.f) || !isfinite(p)) bad |= ST_BAD_PI;
    const double lp = (p > 0.f) ? log((double)p) : -CUDART_INF;
    const double cd = unit ? 0.0 : 1.4426950408889634074 * (lp - 0.5 * slog);
    const double eps = 9.765625e-04 * 1.015625;
    double bnn, c, al, be, numax = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) numax = fmax(numax, fabs(nv[i]));
    numax = (double)(float)warp_max(numax);          // (the value screen_plane_kernel gets)
    bool capped = false;
    for (;;) {                                       // (at most twice; the same way in every lane)
        double absab = 0.0, bmax = 0.0, cmax = 0.0;
        bnn = 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double b = capped ? fmin(bv[i], screen_cap(D, numax)) : bv[i];
            bnn += b * nv[i] * nv[i];
            absab += 2.0 * b * fabs(nv[i]) + b;
            bmax = fmax(bmax, b);
            cmax = fmax(cmax, fmax(b, 2.0 * b * fabs(nv[i])));
        }
        bnn = warp_sum(bnn); absab = warp_sum(absab); bmax = warp_max(bmax); cmax = warp_max(cmax);
        c = cd - bnn;
        al = eps * bnn + 5.9604644775390625e-08 * absab + 2.98023223876953125e-08 * 0.5 * D + 3.814697265625e-06 * fabs(c) + 0.02;
        be = (unit ? 1.0 : 3.0) * eps * bmax + 2.98023223876953125e-08 * 1.5;
        if (unit) {                                  // (a centroid that is too far from the others for 16 bits: the dense kernels)
            if (!(cmax <= 60000.0) || !(bnn < -0.5 * (double)SCR_NEVER)) bad |= ST_NONFINITE;
            break;
        }
        if (capped || !(al + be * D > (double)SCR_SHARP || cmax > 60000.0)) break;
        capped = true;
    }
    if (lane == 0) {
        if (c2) c2[k] = (float)cd;
        c2d[k] = cd;
        const bool on = p > 0.f && isfinite(c) && isfinite(al) && isfinite(be);
        prm[k] = make_float4(on ? (float)c : -CUDART_INF_F, on ? (float)(al * 1.000001) : 0.f, on ? (float)(be * 1.000001) : 0.f, (float)numax);
        key[k] = !on ? CUDART_INF_F : capped ? SCR_CAPPED : (float)(al + be * D);
        if (on) atomicAdd(ctl + SC_ACTIVE, 1);
        // (k-means: the kernels of the dense path say what becomes of it, some report it and some do not)
        if (bad && unit) ctl[SC_DENSE] = 1;
        else if (bad) atomicOr(status, bad);
    }
}

// Whether the screening pays, ahead of the sweep: the exact log-densities of 16 groups of four consecutive rows, spread evenly over
// the call's data so that neither the order of the rows nor one odd region of them decides, and from those how many pairs the sweep
// would mark with its allowances.  Dense are data with more pairs than pay on average, and data of which a 16th or so lies
// together in a region where the pairs of 32 neighbours outgrow their room: those rows would leave the sweep without a list.
// Sixteen CTAs share a group, a 16th of the components each; the last of them to finish counts.  They run beside the CTAs of
// screen_plane_kernel, which take 3 us longer for it.  (Beside the transform of the first piece they cost as much, and broad data its
// time.)  Before, one tile of 256 points above the limit among the first 148 made the whole call dense: 200K x 32, K = 64 with an
// overlapping region at its end took 475 us, of which 180 were the sweep for nothing, now 300 + 55; with the region at its start too.
__device__ __forceinline__ unsigned order_up(float v) { const unsigned b = __float_as_uint(v); return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u); }
__device__ __forceinline__ float order_down(unsigned o) { return __uint_as_float(o ^ ((o >> 31) ? 0x80000000u : 0xffffffffu)); }
struct ProbeArgs {
    ScreenProbe p;
    int K;
    const float *mu, *w2;
    const double* c2d;
    const float4* prm;
    const float* key;
    unsigned* probe;
    int first;               // the first of the probe's CTAs
    float2* bounds;          // [PR_GROUPS * PR_ROWS][K] (a component without a weight: -inf, one without a lower bound: -inf, upper)
    int* ctl;
};
__device__ void screen_probe(const ProbeArgs& a, int D, const float* __restrict__ sd, const float* __restrict__ gd) {
    __shared__ __align__(16) float x_s[PR_ROWS][128];
    __shared__ float nrm_s[PR_ROWS];
    __shared__ int last_s, crowd_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l8 = lane & 7, sub = lane >> 3, K = a.K;
    const int b = (int)blockIdx.x - a.first, grp = b / PR_CTAS, share = (K + PR_CTAS - 1) / PR_CTAS, k0 = min(K, (b % PR_CTAS) * share), k1 = min(K, k0 + share);
    if (tid == 0) crowd_s = 0;
    unsigned* const lower = a.probe + grp * (PR_ROWS + 1);
    float2* const bounds = a.bounds + (size_t)grp * PR_ROWS * K;
    for (int e = tid; e < PR_ROWS * 128; e += 256) {
        const int r = e >> 7, d = e & 127;
        const int64_t row = (int64_t)(((double)grp + 0.5) / PR_GROUPS * (double)a.p.n) + r;
        x_s[r][d] = d < D ? __ldg(a.p.X + (row < a.p.n ? row : a.p.n - 1) * D + d) : 0.f;
    }
    __syncthreads();
    if (warp < PR_ROWS) {                            // warp = row
        float q = 0.f;
        for (int d = lane; d < D; d += 32) { const float u = (x_s[warp][d] - __ldg(gd + d)) * __ldg(sd + d); q = fmaf(u, u, q); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (lane == 0) nrm_s[warp] = q;
    }
    __syncthreads();
    // eight lanes per component; lane l8 < PR_ROWS then holds its value for row l8
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(a.mu) & 15) == 0);      // (w2: scratch, aligned)
    const float nrm = nrm_s[l8 % PR_ROWS];
    float low = -CUDART_INF_F;
    for (int kb = k0 + warp * 4; kb < k1; kb += 32) {
        const int k = min(kb + sub, k1 - 1);
        const float *m = a.mu + (size_t)k * D, *w = a.w2 + (size_t)k * D;
        const float4 e = __ldg(a.prm + k);
        const float c = (float)__ldg(a.c2d + k), key = __ldg(a.key + k);
        float q[PR_ROWS];
#pragma unroll
        for (int r = 0; r < PR_ROWS; ++r) q[r] = 0.f;
        if (vec) {
            float4 mv[4], wv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int d = 4 * (l8 + 8 * i);
                mv[i] = wv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (d < D) { mv[i] = __ldg(reinterpret_cast<const float4*>(m + d)); wv[i] = __ldg(reinterpret_cast<const float4*>(w + d)); }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int r = 0; r < PR_ROWS; ++r) {
                    const float4 x = *reinterpret_cast<const float4*>(&x_s[r][4 * (l8 + 8 * i)]);
                    const float t0 = x.x - mv[i].x, t1 = x.y - mv[i].y, t2 = x.z - mv[i].z, t3 = x.w - mv[i].w;
                    q[r] = fmaf(wv[i].x * t0, t0, q[r]); q[r] = fmaf(wv[i].y * t1, t1, q[r]);
                    q[r] = fmaf(wv[i].z * t2, t2, q[r]); q[r] = fmaf(wv[i].w * t3, t3, q[r]);
                }
        } else {
            for (int d = l8; d < D; d += 8) {
                const float mv = __ldg(m + d), wv = __ldg(w + d);
#pragma unroll
                for (int r = 0; r < PR_ROWS; ++r) { const float t = x_s[r][d] - mv; q[r] = fmaf(wv * t, t, q[r]); }
            }
        }
        float mine = 0.f;
#pragma unroll
        for (int r = 0; r < PR_ROWS; ++r) {
            q[r] += __shfl_xor_sync(0xffffffffu, q[r], 1);
            q[r] += __shfl_xor_sync(0xffffffffu, q[r], 2);
            q[r] += __shfl_xor_sync(0xffffffffu, q[r], 4);
            if (l8 == r) mine = q[r];
        }
        if (kb + sub < k1 && l8 < PR_ROWS) {
            const float l = c - mine, E = fmaf(e.z, nrm, e.y);
            const bool on = e.x > -CUDART_INF_F;
            const float2 at = make_float2(on && key < SCR_CAPPED ? l - E : -CUDART_INF_F, on ? l + E : -CUDART_INF_F);
            bounds[(size_t)l8 * K + k] = at;
            low = fmaxf(low, at.x);
        }
    }
    low = fmaxf(low, __shfl_xor_sync(0xffffffffu, low, 8));
    low = fmaxf(low, __shfl_xor_sync(0xffffffffu, low, 16));
    if (sub == 0 && l8 < PR_ROWS) atomicMax(lower + l8, order_up(low));
    __threadfence();
    __syncthreads();
    if (tid == 0) last_s = atomicAdd(lower + PR_ROWS, 1u) == PR_CTAS - 1;
    __syncthreads();
    if (!last_s || warp >= PR_ROWS) return;
    __threadfence();
    const float2* mine = bounds + (size_t)warp * K;                          // warp = row
    float cut = order_down(__ldcg(lower + warp)) - a.p.margin;
    if (a.p.top > 1) {                                 // the sweep's bound for the `top` largest: the largest lower bounds of eights of components
        float best[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll 4
        for (int k0 = lane * 8; k0 < K; k0 += 256) {
            float x = -CUDART_INF_F;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (k0 + j < K) x = fmaxf(x, __ldcg(mine + k0 + j).x);
#pragma unroll
            for (int j = 0; j < 4; ++j) { const float keep = fmaxf(best[j], x); x = fminf(best[j], x); best[j] = keep; }
        }
        float m = 0.f;
        for (int r = 0; r < a.p.top; ++r) {
            m = best[0];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == __ffs(__ballot_sync(0xffffffffu, best[0] == m)) - 1) { best[0] = best[1]; best[1] = best[2]; best[2] = best[3]; best[3] = -CUDART_INF_F; }
        }
        cut = fminf(cut, m);
    }
    cut = fmaxf(cut, 0.5f * SCR_NEVER);
    int cnt = 0;
#pragma unroll 16
    for (int k = lane; k < K; k += 32) cnt += __ldcg(mine + k).y >= cut ? 1 : 0;
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    // (a quarter more than the sweep's limit: a sample.  The sums only grow, so whoever takes one across its limit says so.)
    if (lane == 0 && ((float)(atomicAdd(a.ctl + SC_PROBED, cnt) + cnt) > 1.25f * a.p.max_marks * (PR_GROUPS * PR_ROWS) ||
                      (atomicAdd(&crowd_s, cnt) + cnt > SCR_SLOTS * PR_ROWS && a.p.max_marks <= SCR_SLOTS)))
        a.ctl[SC_DENSE] = 1;
}

// Where dimension d stands in the contraction: chunk c of the KS chunks of eight has dimensions 4 c .. 4 c + 3 and 4 (KS + c) .. + 3, so
// that neighbouring lanes that form one chunk each read neighbouring 16 bytes of a row.
__host__ __device__ __forceinline__ int screen_slot(int d, int KS) { return d < 4 * KS ? (d >> 2) * 8 + (d & 3) : ((d - 4 * KS) >> 2) * 8 + 4 + (d & 3); }
constexpr int SW_CSLOT = 4096;               // a group's constants: 128 rows of 16 halves
// Positions of the components in the sweep: ascending by the allowance of a typical point, so that 32 neighbours, which are
// screened with the largest allowance among them, have similar ones (the capped components come last).  A warp per component:
// its rank among the keys is its position, and it writes its own row (a sort of the keys in every CTA took 20 us).  The
// coefficients are written as the sweep has them in shared memory (screen_group_bytes per group of 128 positions: the constants,
// then the atoms of 32 dimensions, swizzled), so that a stage is one contiguous copy.
__global__ void __launch_bounds__(256) screen_plane_kernel(const ProbeArgs probe, int D, int K, int Kpad, int unit, const float* __restrict__ mu,
                                                           const float* __restrict__ w2, const float* __restrict__ sd,
                                                           const float* __restrict__ gd, const float4* __restrict__ prm,
                                                           const float* __restrict__ key, unsigned char* __restrict__ img,
                                                           int4* __restrict__ blk, int* __restrict__ comp_of) {
    if ((int)blockIdx.x >= probe.first) {
        screen_probe(probe, D, sd, gd);
        return;
    }
    const int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    int pos = k;
    bool on = false, capped = false;
    float4 q = make_float4(-CUDART_INF_F, 0.f, 0.f, 0.f);
    // (capped components and those without a weight at the far end, what is left of Kpad between them and the others: a block that
    // holds a capped component has no lower bound)
    if (k >= K) {
        int before = 0;
        for (int j = lane; j < K; j += 32) before += __ldg(key + j) < SCR_CAPPED ? 1 : 0;
        pos = __reduce_add_sync(0xffffffffu, before) + k - K;
    } else {
        const float mine = __ldg(key + k);
        int before = 0;
#pragma unroll 8
        for (int j = lane; j < K; j += 32) {
            const float o = __ldg(key + j);
            before += (o < mine || (o == mine && j < k)) ? 1 : 0;
        }
        pos = __reduce_add_sync(0xffffffffu, before) + (mine >= SCR_CAPPED ? Kpad - K : 0);
        on = mine < CUDART_INF_F;
        capped = on && mine >= SCR_CAPPED;
        if (on) q = __ldg(prm + k);
    }
    const int r = pos & 127;
    unsigned char* grp = img + (size_t)(pos >> 7) * screen_group_bytes(D, unit != 0);
    const int nch = (D + 7) / 8, ndim = unit ? (nch + 1) / 2 * 16 : nch * 8;     // (unit: a k-step holds two chunks of u)
    for (int d = lane; d < ndim; d += 32) {                  // (in the order of screen_slot; beyond D: zeros)
        float a = 0.f, b = 0.f;
        if (on && d < D) {
            const float s = __ldg(sd + d);
            double bd = (double)__ldg(w2 + (size_t)k * D + d) / ((double)s * (double)s);
            if (capped) bd = fmin(bd, screen_cap(D, (double)q.w));
            const double nu = ((double)__ldg(mu + (size_t)k * D + d) - (double)__ldg(gd + d)) * (double)s;
            a = (float)(2.0 * bd * nu);
            b = (float)(-bd);
        }
        // k-step d / 8 holds eight dimensions of u and the same eight of u^2: two 16-byte chunks of a 128-byte row, swizzled
        const int z = d < 8 * nch ? screen_slot(d, nch) : d;
        if (unit) {
            *reinterpret_cast<__half*>(grp + SW_CSLOT + (z >> 6) * 16384 + r * 128 + ((((z >> 3) & 7) ^ (r & 7)) << 4) + 2 * (z & 7)) = __float2half_rn(a);
            continue;
        }
        unsigned char* o = grp + SW_CSLOT + (z >> 5) * 16384 + r * 128;
        const int c = 2 * ((z >> 3) & 3);
        *reinterpret_cast<__half*>(o + ((c ^ (r & 7)) << 4) + 2 * (z & 7)) = __float2half_rn(a);
        *reinterpret_cast<__half*>(o + (((c + 1) ^ (r & 7)) << 4) + 2 * (z & 7)) = __float2half_rn(b);
    }
    if (lane == 0) {
        comp_of[pos] = on ? k : -1;
        const float c = fmaxf(q.x, SCR_NEVER);                // (no weight: no mark)
        const __half h1 = __float2half_rn(c / 256.f);
        const float r1 = c - 256.f * __half2float(h1);
        const __half h2 = __float2half_rn(r1), h3 = __float2half_rn(r1 - __half2float(h2));
        uint4* pc = reinterpret_cast<uint4*>(grp) + 2 * r;
        const int sw = (r >> 2) & 1;
        pc[sw] = make_uint4((uint32_t)__half_as_ushort(h1) | ((uint32_t)__half_as_ushort(h2) << 16), __half_as_ushort(h3), 0u, 0u);
        pc[sw ^ 1] = make_uint4(0u, 0u, 0u, 0u);
        // the largest allowances of the block of 32 positions (non-negative floats order as integers), and whether it holds a
        // capped component (then it has no lower bound)
        int* bk = reinterpret_cast<int*>(blk + (pos >> 5));
        atomicMax(bk, __float_as_int(q.y));
        atomicMax(bk + 1, __float_as_int(q.z));
        if (capped) bk[2] = 1;
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Rows of u in shared memory: `chunks` 16-byte chunks (8 dimensions each).  Chunk c of row r sits at place screen_place(c, r): the
// sweep reads a row per lane, and eight neighbouring rows' chunks c then lie in different banks.
__host__ __device__ __forceinline__ int screen_chunks(int D) { return D <= 32 ? 4 : D <= 64 ? 8 : 16; }
__device__ __forceinline__ int screen_place(int c, int row, int chunks) { return chunks == 4 ? c ^ ((row >> 1) & 3) : c ^ (row & 7); }

// X -> fp16 plane of u and |u|^2, for the shapes that the sweep does not convert itself.  L lanes per row, 8 dimensions each.  Bound by
// memory: 4 D bytes in, 2 D out.  Data that are not finite are left to the dense kernels: what becomes of them differs from entry point to entry point
// and from path to path.
template <int L>
__global__ void __launch_bounds__(256) screen_transform_kernel(const float* __restrict__ X, int64_t n, int D, int chunks, const float* __restrict__ sd,
                                                               const float* __restrict__ gd, unsigned char* __restrict__ y,
                                                               float* __restrict__ n2, int* __restrict__ ctl) {
    if (screen_off(ctl)) return;
    const bool vec_ok = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    const int l = threadIdx.x % L, KS = (D + 7) / 8;
    auto dim = [&](int j) { return l < KS ? (j < 4 ? 4 * l + j : 4 * (KS + l) + j - 4) : D; };       // (see screen_slot)
    constexpr int RPB = 256 / L;
    float gv[8], sv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { gv[j] = dim(j) < D ? __ldg(gd + dim(j)) : 0.f; sv[j] = dim(j) < D ? __ldg(sd + dim(j)) : 0.f; }
    bool bad = false;
    const int64_t step = (int64_t)gridDim.x * RPB;
    auto load = [&](int64_t row, float (&x)[8]) {
        if (row < n && vec_ok && dim(7) < D) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(X + row * D + dim(0))), b = __ldg(reinterpret_cast<const float4*>(X + row * D + dim(4)));
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = (row < n && dim(j) < D) ? __ldg(X + row * D + dim(j)) : 0.f;
        }
    };
    auto store = [&](int64_t row, const float (&x)[8]) {
        float nrm = 0.f;
        bool far = false;
        uint32_t xh[4];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            bad |= !(fabsf(x[j]) <= 3.0e38f) || !(fabsf(x[j + 1]) <= 3.0e38f);
            float u0 = (x[j] - gv[j]) * sv[j], u1 = (x[j + 1] - gv[j + 1]) * sv[j + 1];       // (beyond D: zeros)
            far |= !(fabsf(u0) <= 240.f) || !(fabsf(u1) <= 240.f);
            u0 = fminf(fmaxf(u0, -240.f), 240.f);
            u1 = fminf(fmaxf(u1, -240.f), 240.f);
            nrm = fmaf(u0, u0, fmaf(u1, u1, nrm));
            const __half2 h = __floats2half2_rn(u0, u1);
            xh[j / 2] = *reinterpret_cast<const uint32_t*>(&h);
        }
        if (far) nrm = CUDART_INF_F;                 // (a clamped coordinate: no bound holds, the row is evaluated in full)
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        if (row >= n) return;
        if (l < KS) *reinterpret_cast<uint4*>(y + ((size_t)row * chunks + screen_place(l, (int)row, chunks)) * 16) = make_uint4(xh[0], xh[1], xh[2], xh[3]);
        if (l == 0) n2[row] = nrm * 1.0001f;
    };
    // (every lane of a warp takes the same number of steps: the row sums are shuffles; two rows' loads in flight)
    for (int64_t r0 = (int64_t)blockIdx.x * RPB; r0 < n; r0 += 2 * step) {
        const int64_t row = r0 + threadIdx.x / L;
        float xa[8], xb[8];
        load(row, xa);
        load(row + step, xb);
        store(row, xa);
        store(row + step, xb);
    }
    if (bad) ctl[SC_DENSE] = 1;
}

// ------------------------------------------------------------------------------------------------------------------
// Sweep
constexpr int SW_PSLOT = 32768;              // a coefficient stage: two atoms of 128 components
constexpr int SW_REGS = 168, SW_REGS_FEW = 88;       // CONVERT: of a softmax thread and of the others: (168 + 88) x 256 = what 512 threads have at launch
constexpr int SW_XBYTES = 16384 + 32;        // CONVERT: a chunk of X, from the 16-byte boundary before it on
// Where the points' rows come from.  CONVERT: X itself, converted by four warps of the sweep.  Otherwise screen_transform_kernel has
// written the rows of u (16-bit), which come by bulk copy.
template <bool CONVERT>
struct Sweep {
    static constexpr int THREADS = CONVERT ? 512 : 352;      // 8 softmax warps, 4 that convert, producer warp, an MMA warp per half of the tile, a warp that fetches X
    static constexpr int CONVERTER = 8, PRODUCER = CONVERT ? 12 : 8, MMA = PRODUCER + 1, FETCH = 15;
    static constexpr int PS = CONVERT ? 3 : 4;               // coefficient stages
    static constexpr int CSLOTS = CONVERT ? 3 : 4;           // groups in flight that have constants: as many as there are stages, of which a group takes one or two
    static constexpr int ENT = CONVERT ? 7 : 10;             // blocks of 32 components a point can have marks in: in shared memory,
    static constexpr int SPILL = 32 - ENT;                   // and, rarely needed, in global memory (a mask has 32 bits)
    static constexpr int UOFF = PS * SW_PSLOT;               // the next tile's rows of u (256 x 16 chunks bytes; not CONVERT: 8 chunks at most)
    static constexpr int COFF = UOFF + (CONVERT ? 65536 : 32768);                // constants of the groups in flight
    static constexpr int AOFF = COFF + CSLOTS * SW_CSLOT;    // the points' side of the constants: 128 rows (256, 1, 1, 0, ...)
    static constexpr int EOFF = AOFF + 4096;
    static constexpr int TOFF = EOFF + ENT * 256 * 8;        // allowances of every block
    static constexpr int NOFF = TOFF + SCR_MAX_K / 32 * 8;   // CONVERT: |u|^2 of the next tile's rows, chunks of X
    static constexpr int XOFF = NOFF + (CONVERT ? 256 * 4 : 0);
    static constexpr int BOFF = XOFF + (CONVERT ? 2 * SW_XBYTES : 0);
    static constexpr int SMEM = BOFF + 256 + 1024;
    enum { PFULL = 0, PEMPTY = PFULL + PS, UFULL = PEMPTY + PS, UEMPTY, AFULL, LFULL = AFULL + 2, LEMPTY = LFULL + 2, FINAL = LEMPTY + 2, XFULL = FINAL + 2,
           XEMPTY = XFULL + 2, COUNT = XEMPTY + 2 };
    static_assert(COUNT * 8 <= 256, "barriers");
    static_assert(!CONVERT || (CONVERTER % 4 == 0 && THREADS % 128 == 0 && (SW_REGS * CONVERTER + SW_REGS_FEW * (THREADS / 32 - CONVERTER)) * 32 <= 65536), "registers of whole warpgroups");
    static_assert(SMEM <= 232448, "shared memory");
    static_assert(SPILL <= SCR_SPILL, "room for the spilled entries");
};
// Which way pays.  The line was drawn by the sweep of steps, per 1.02M points (us, converted by the sweep / sweep + transform; K = 256, 1024,
// 4096): D = 128: 238 / 264, 442 / 534, 1468 / 1603; D = 80 (K = 256, 4096): 240 / 282, 1242 / 1420; D = 64: 141 / 170, 334 / 350, 1029 / 950;
// D = 48: 143 / 185, 359 / 359, 1103 / 1025; D = 32: 114 / 129, 358 / 300, 1161 / 1082; D = 16 (K = 256): 102 / 113.  The transform costs about
// 1.06 us per dimension; the converting warps cost the softmax warps issue slots and instruction cache, which matters where the MMAs are
// short.  Whole calls with the roles' loops as they are now: steps 64 x 512 836 / 809, 64 x 1024 938 / 944, 48 x 1024 1052 / 1022, 32 x 1024
// 966 / 908.  Half the contraction (k-means) and two passes (top-2) would put the line a little elsewhere: k-means 64 x 1024 620 / 660,
// 32 x 1024 558 / 565, 32 x 4096 1226 / 1164; top-2 48 x 1024 1051 / 1079, 64 x 1024 1046 / 1022, 64 x 4096 2597 / 2362.
inline bool screen_converts(int D, int K) { return D > 64 || (D > 32 && K <= 512) || K <= 256; }

// two fp32 operations per instruction
__device__ __forceinline__ uint64_t pack2(uint32_t a, uint32_t b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ float lo2(uint64_t a) { return __uint_as_float((uint32_t)a); }
__device__ __forceinline__ float hi2(uint64_t a) { return __uint_as_float((uint32_t)(a >> 32)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { return fma2(b, 0xBF800000BF800000ull, a); }      // (a - b, rounded once)
// Operand of one k-step: rows of 32 bytes, 32-byte swizzle, groups of eight rows 256 bytes apart.
__device__ __forceinline__ uint64_t make_desc32(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(256 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}
// The wait for a load of accumulators that is in flight while others are worked on: its registers go through the wait, so that
// nothing that uses them can be placed before it.
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), 
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), 
                 "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]), 
                 "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31]) :: "memory");
}
__device__ __forceinline__ float max3(float a, float b, float c) { float r; asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }

struct SweepParams {
    int64_t n;
    int KA, KS, NG;          // atoms and k-steps of the contraction, groups of 128 components
    int KC;                  // chunks of eight dimensions: a k-step has one and its squares, or (unit) two
    int chunks;              // 16-byte chunks that a row of u takes
    bool unit;
    const float* X;
    int D;
    const float *sd, *gd;
    const unsigned char* y;  // (not CONVERT: rows of u, |u|^2)
    const float* n2;
    const unsigned char* img;
    int gbytes;              // of the image of a group
    float margin;
    const int4* blk;
    unsigned* pt_off;
    int* pt_cnt;
    uint2* words;
    unsigned long long* spill;
    int* ovf;
    int* ctl;
    int* status;
    int test_silent;                // >= 0: that CTA keeps back the news of its first products (time-out test)
};

// The points' way into the sweep: rows of X through a ring of two slots of 16 KB, which a warp of its own fills by untiled bulk copies,
// and from there, by four converting warps, as rows of u (and |u|^2) into shared memory.  A copy starts at the 16-byte boundary
// before its first byte and ends at the one behind its last, so that any X will do; what would reach beyond X's own bytes is read
// with plain loads.  A chunk has 512 / L rows, L = 2^SH lanes of eight dimensions per row, four rows per lane.  One warp per scheduler
// has nothing to hide its latencies behind but its own instructions, so each chunk's fixed cost counts: with 2 KB per warp and copy,
// requested by the warps themselves, a chunk took 1700 cycles (180 to see that it is there, 500 to ask for the next, 700 to convert it)
// and the sweep waited for them.
// bar_wait for those who mostly wait (the hint lets the hardware keep them away from the scheduler for longer).
__device__ __forceinline__ bool bar_wait_idle(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status) {
    for (int it = 0; it < 4; ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                     : "=r"(ok) : "r"(bar), "r"(parity), "r"(5000) : "memory");
        if (ok) return true;
        if (*abort_flag) return false;
    }
    return bar_wait(bar, parity, abort_flag, status, false);
}
struct SweepRows {
    uint64_t xb;                 // the 16-byte boundary at or before X; offsets below count from it (at most 2^20 rows of 512 bytes)
    uint32_t shift, D4, end;
    int n, R, per, tstep, first;
    __device__ __forceinline__ SweepRows(const SweepParams& p, int sh) {
        const uint64_t x = reinterpret_cast<uint64_t>(p.X);
        xb = x & ~(uint64_t)15;
        shift = (uint32_t)(x & 15u);
        D4 = 4u * (uint32_t)p.D;
        n = (int)p.n;
        end = shift + (uint32_t)n * D4;
        R = 512 >> sh;
        per = 1 << (sh - 1);                                 // chunks per tile
        first = (int)blockIdx.x * SCR_TILE;
        tstep = (int)gridDim.x * SCR_TILE;
    }
    // whether the chunk from `row` on comes by bulk copy
    __device__ __forceinline__ bool range(int row, uint32_t& lo, uint32_t& bytes) const {
        const uint32_t q = shift + (uint32_t)row * D4, hi = (q + (uint32_t)R * D4 + 15u) & ~15u;
        lo = q & ~15u;
        bytes = hi - lo;
        return row + R <= n && lo >= shift && hi <= end;
    }
};
__device__ __forceinline__ int screen_lane_shift(int KC) { return KC > 8 ? 4 : KC > 4 ? 3 : KC > 2 ? 2 : 1; }

template <int SH>
__device__ __forceinline__ void screen_convert(const SweepParams& p, unsigned char* smem, int cw, int lane, int ntl, volatile int* abort_flag) {
    constexpr int L = 1 << SH, RW = 32 >> SH;                // rows per warp and step
    using S = Sweep<true>;
    const SweepRows rows(p, SH);
    const int D = p.D, l = lane & (L - 1), sub = lane >> SH;
    const int d0 = 4 * l, d1 = 4 * (p.KC + l);               // dimensions of this lane: d0 .. d0 + 3 and d1 .. d1 + 3 (see screen_slot)
    const bool on = l < p.KC;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::BOFF);
    float* nrm_s = reinterpret_cast<float*>(smem + S::NOFF);
    const bool vec = ((D & 3) == 0) && rows.shift == 0, in0 = on && d0 < D, in1 = on && d1 < D;
    uint64_t s2[4], g2[4];                                   // u = s x - s g: s a power of two, so the same as s (x - g)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int d = j < 2 ? d0 + 2 * j : d1 + 2 * j - 4;
        const bool a = on && d < D, b = on && d + 1 < D;     // (a lane without a chunk adds nothing to |u|^2)
        const float sa = a ? __ldg(p.sd + d) : 0.f, sb = b ? __ldg(p.sd + d + 1) : 0.f;
        s2[j] = pack2(__float_as_uint(sa), __float_as_uint(sb));
        g2[j] = pack2(__float_as_uint(a ? -sa * __ldg(p.gd + d) : 0.f), __float_as_uint(b ? -sb * __ldg(p.gd + d + 1) : 0.f));
    }
    // where this lane's 16 bytes of u go: row r0 + 4 RW h of a tile, r0 = cw RW + sub + 128 k (SH = 4: 32 k)
    const int rl = cw * RW + sub;
    uint32_t c = 0;
    bool ok = true;
    for (int i = 0; i < ntl && ok; ++i) {
        int row0 = rows.first + i * rows.tstep;
#pragma unroll 1
        for (int k = 0; k < rows.per; ++k, ++c, row0 += rows.R) {
            const uint32_t slot = c & 1u;
            ok = __all_sync(0xffffffffu, bar_wait_idle(smem_u32(&bars[S::XFULL + slot]), (c >> 1) & 1u, abort_flag, p.status));
            if (!ok) break;
            uint32_t lo, bytes;
            uint64_t x[4][4];
            if (rows.range(row0, lo, bytes)) {
                const unsigned char* src = smem + S::XOFF + slot * SW_XBYTES + (rows.shift + (uint32_t)row0 * rows.D4 - lo) + (uint32_t)rl * rows.D4;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const unsigned char* q = src + (uint32_t)(h * 4 * RW) * rows.D4;
                    if (vec) {
                        ulonglong2 a = make_ulonglong2(0ull, 0ull), b = a;
                        if (in0) a = *reinterpret_cast<const ulonglong2*>(q + 4 * d0);
                        if (in1) b = *reinterpret_cast<const ulonglong2*>(q + 4 * d1);
                        x[h][0] = a.x; x[h][1] = a.y; x[h][2] = b.x; x[h][3] = b.y;
                    } else {
                        const uint32_t* w = reinterpret_cast<const uint32_t*>(q);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int d = j < 2 ? d0 + 2 * j : d1 + 2 * j - 4;
                            x[h][j] = pack2(on && d < D ? w[d] : 0u, on && d + 1 < D ? w[d + 1] : 0u);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int row = row0 + rl + h * 4 * RW;
                    const float* q = p.X + (int64_t)row * D;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int d = j < 2 ? d0 + 2 * j : d1 + 2 * j - 4;
                        x[h][j] = pack2(row < rows.n && on && d < D ? __float_as_uint(__ldg(q + d)) : 0u,
                                        row < rows.n && on && d + 1 < D ? __float_as_uint(__ldg(q + d + 1)) : 0u);
                    }
                }
            }
            __syncwarp();                                    // (the warp's part of the slot has been read)
            if (lane == 0) bar_arrive(smem_u32(&bars[S::XEMPTY + slot]));
            if (k == 0 && i > 0)                             // the rows of the tile before have been taken
                ok = __all_sync(0xffffffffu, bar_wait_idle(smem_u32(&bars[S::UEMPTY]), (uint32_t)((i - 1) & 1), abort_flag, p.status));
            if (!ok) break;
            float nrm[4];
            const int r0 = k * rows.R + rl;                  // of the tile
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int r = r0 + h * 4 * RW;
                uint64_t u[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) u[j] = fma2(x[h][j], s2[j], g2[j]);
                const uint64_t a = add2(fma2(u[2], u[2], mul2(u[0], u[0])), fma2(u[3], u[3], mul2(u[1], u[1])));
                nrm[h] = lo2(a) + hi2(a);
                if (!(nrm[h] <= 57600.f)) {                  // (a coordinate beyond 240, or one that is not finite?)
                    bool bad = false, far = false;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        bad |= !(fabsf(lo2(x[h][j])) <= 3.0e38f) || !(fabsf(hi2(x[h][j])) <= 3.0e38f);
                        far |= !(fabsf(lo2(u[j])) <= 240.f) || !(fabsf(hi2(u[j])) <= 240.f);
                        u[j] = pack2(__float_as_uint(fminf(fmaxf(lo2(u[j]), -240.f), 240.f)), __float_as_uint(fminf(fmaxf(hi2(u[j]), -240.f), 240.f)));
                    }
                    if (bad) p.ctl[SC_DENSE] = 1;            // (data that are not finite are left to the dense kernels: what becomes of
                    if (far) nrm[h] = CUDART_INF_F;          // them differs from path to path; a clamped coordinate: no bound holds, the row
                }                                            // is evaluated in full)
                if (on) {
                    uint32_t xh[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const __half2 hh = __floats2half2_rn(lo2(u[j]), hi2(u[j]));
                        xh[j] = *reinterpret_cast<const uint32_t*>(&hh);
                    }
                    *reinterpret_cast<uint4*>(smem + S::UOFF + (r * p.chunks + screen_place(l, r, p.chunks)) * 16) = make_uint4(xh[0], xh[1], xh[2], xh[3]);
                }
            }
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
                for (int h = 0; h < 4; ++h) nrm[h] += __shfl_xor_sync(0xffffffffu, nrm[h], o);
            if (l == 0) {
#pragma unroll
                for (int h = 0; h < 4; ++h) nrm_s[r0 + h * 4 * RW] = nrm[h] * 1.0001f;
            }
        }
        if (ok) bar_arrive(smem_u32(&bars[S::UFULL]));
    }
}

// Tile = 256 points in two halves of 128 TMEM lanes, a thread per point.  The points' operand [u | u^2] lives in TENSOR MEMORY
// (columns 256 + 128 h of half h; the squares are formed when it is written), so that shared memory has only the coefficients to
// deliver: with both operands there its bandwidth alone (8 KB per MMA of 64 cycles, besides the incoming stages) held the sweep to
// half the tensor cores' rate.  Coefficients come as 1-D bulk copies of an image that screen_plane_kernel laid out swizzled, in
// stages of 32 KB.  Per group of 128 components the tensor cores form half 0 (columns 0-127) and half 1 (128-255) from the same
// stages; a group's constants are one more product, of 16 columns.  A group's accumulators go into registers at once (128 of
// them), so that the next group of the half is formed while they are worked through: the four blocks' maxima first, then their marks.  When
// the last group of a tile has been formed, the half's operand is replaced by the next tile's rows, which wait in shared memory,
// before those accumulators are read.
// MMA time per group: 2 x (ceil(D / 8) + 1) x 64.5 cycles; a group takes 2600 at D = 128 with 32 of them, a tile about 3000 more for its
// list and the next one's operand, at the 1.65 to 1.75 GHz that the power limit leaves (27 tiles per CTA, K = 1024, not converting: 383 to 402 us
// at D = 128, 261 to 282 at D = 64, where the softmax threads set the pace; block by block, each one's marks before the next one's
// maxima: 400, 318).  Converting, the tensor cores are busy 59 % of the time instead of 69 %: the converting warps' instructions.  Pairs of
// CTAs (cta_group::2, half the coefficients each) wait for each other's softmax threads: 550 us against 459 then.
//
// TOP: how many of a point's largest values are wanted for certain.  1: everything within the margin of the largest.  More (the top-m
// assignment): also everything that could be among the TOP largest.  The bound for those is the TOP-th largest of the lower bounds of
// the quarters of every block: different components, so the TOP-th largest value cannot be below it.  It rises as the sweep goes on, most of
// all in the first group, under whose bounds twice as many pairs were marked as the final one leaves.  So the first group passes
// once more at the end and is marked then, the others as they come: emulated on the clusters of 128 x 1024 3.13 marks per point, as many as
// with all components twice (5.6 in one pass; top-4 12.6, 16.8).  1.02M points, top-2 (us): 128 x 1024 1270 -> 955, 32 x 1024 941 -> 806,
// 64 x 4096 2447 -> 1679, 128 x 4096 3723 -> 2333.
template <int TOP, bool CONVERT>
__global__ void __launch_bounds__(Sweep<CONVERT>::THREADS, 1)
screen_sweep_kernel(const SweepParams p) {
    using S = Sweep<CONVERT>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, drain_s;
    if (screen_off(p.ctl)) return;
    volatile int* abort_flag = &abort_s;
    volatile int* drain_flag = &drain_s;
    // (role: the warp's number, uniform for the compiler too, by which the last warpgroup's roles part.  By `warp` each of their loops carries the
    // bookkeeping of branches that lanes could take one by one: 3M points, 72 x 1024, log-densities 2113 -> 1975 us, k-means of 128 x 1024 1991 -> 1867.
    // The other warpgroups have one role each and keep `warp`: top-2 of 1M x 128, K = 1024 1395 us, with `role` for all 1417.)
    const int tid = threadIdx.x, warp = tid >> 5, role = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int64_t ntiles = (p.n + SCR_TILE - 1) / SCR_TILE;
    const int64_t ntl = ((int64_t)blockIdx.x < ntiles) ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    const int NG = p.NG, GT = TOP > 1 ? NG + 1 : NG;         // groups of a tile (TOP > 1: the first one twice)
    const int spg = (p.KA + 1) >> 1;              // stages per group
    unsigned char* cons = smem + S::COFF;                    // [CSLOTS][4096]
    float* nrm_s = reinterpret_cast<float*>(smem + S::NOFF);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::BOFF);
    auto BAR = [&](int i) { return smem_u32(&bars[i]); };
    if (tid == 0) {
        abort_s = 0;
        drain_s = 0;
        for (int i = 0; i < S::COUNT; ++i) {
            const bool wg = (i >= S::AFULL && i < S::AFULL + 2) || (i >= S::LEMPTY && i < S::LEMPTY + 2);
            const bool both = i >= S::PEMPTY && i < S::PEMPTY + S::PS;           // (released by the MMA warps of both halves)
            bar_init(BAR(i), i == S::UEMPTY ? 256 : (wg || (CONVERT && i == S::UFULL)) ? 128 : (i == S::XEMPTY || i == S::XEMPTY + 1) ? 4 : both ? 2 : 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == S::MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid < NG * 4) {
        const int4 q = __ldg(p.blk + tid);
        reinterpret_cast<float2*>(smem + S::TOFF)[tid] = make_float2(q.z ? -__int_as_float(q.x) : __int_as_float(q.x), __int_as_float(q.y));      // (sign: no lower bound)
    }
    if (tid < 256) {                                         // rows of 32 bytes, 32-byte swizzle (16-byte chunk ^ bit 2 of the row)
        const int r = tid >> 1, c = (tid & 1) ^ ((r >> 2) & 1);
        reinterpret_cast<uint4*>(smem + S::AOFF)[tid] = c == 0 ? make_uint4(0x3C005C00u, 0x00003C00u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_base_s;

    // The warpgroups of the softmax warps (0 to 7) take the registers that the converting warps (8 to 11) and the last warpgroup give.  A warpgroup
    // executes one instruction, so the last one, which has three roles, does so in the condition ahead of them.  (One for both of those
    // warpgroups, ahead of the converting warps' branch: three registers more than there are, 12 bytes of spills.)
    auto give_registers = [&]() { if (CONVERT) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SW_REGS_FEW)); };
    if (warp < S::CONVERTER) {
        // =========================== softmax warps: thread = TMEM lane = point ===========================
        if (CONVERT) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(SW_REGS));
        const int half = warp >> 2;
        const uint32_t lane_addr = ((uint32_t)((warp & 3) * 32)) << 16;
        const uint32_t col = tmem + half * 128 + lane_addr, acol = tmem + 256 + half * 128 + lane_addr;
        unsigned long long* ent_s = reinterpret_cast<unsigned long long*>(smem + S::EOFF) + tid;
        unsigned long long* ent_g = p.spill + (size_t)blockIdx.x * 256 * S::SPILL + tid;
        // (CONVERT: rows of at most 8 chunks leave half of their buffer to further entries)
        unsigned long long* ent_x = reinterpret_cast<unsigned long long*>(smem + S::UOFF + 32768) + tid;
        const int near_e = CONVERT && p.chunks <= 8 ? S::ENT + 16 : S::ENT;
        auto ent = [&](int e) -> unsigned long long& { return e < S::ENT ? ent_s[256 * e] : e < near_e ? ent_x[256 * (e - S::ENT)] : ent_g[256 * (e - S::ENT)]; };
        const uint4* urow = reinterpret_cast<const uint4*>(smem + S::UOFF) + (size_t)tid * p.chunks;
        uint32_t gi = 0;                                     // groups processed (all tiles)
        int marks = 0;
        const float2* blk = reinterpret_cast<const float2*>(smem + S::TOFF);
        float nrm_next = 0.f;                                // |u|^2 of the row that was taken last
        // this thread's row of tile i (in shared memory) -> the half's operand in tensor memory
        auto operand = [&](int64_t i) {
            const bool got = bar_wait(BAR(S::UFULL), (uint32_t)(i & 1), abort_flag, p.status, false);
            if (__all_sync(0xffffffffu, got)) {
#pragma unroll 1
                for (int q = 0; q < p.KC; q += 8) {          // (eight chunks' loads in flight)
                    uint4 v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        v[j] = (q + j < p.KC) ? urow[screen_place(q + j, tid, p.chunks)] : make_uint4(0u, 0u, 0u, 0u);
                    if (p.unit) {                            // u alone
                        uint32_t w[32];
#pragma unroll
                        for (int j = 0; j < 8; ++j) { w[4 * j] = v[j].x; w[4 * j + 1] = v[j].y; w[4 * j + 2] = v[j].z; w[4 * j + 3] = v[j].w; }
                        tmem_st32(acol + (q >> 3) * 32, w);
                        continue;
                    }
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        uint32_t w[32];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t q[4] = {v[4 * y + j].x, v[4 * y + j].y, v[4 * y + j].z, v[4 * y + j].w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const __half2 h = *reinterpret_cast<const __half2*>(&q[e]);
                                const __half2 sq = __hmul2(h, h);
                                w[8 * j + e] = q[e];
                                w[8 * j + 4 + e] = *reinterpret_cast<const uint32_t*>(&sq);
                            }
                        }
                        tmem_st32(acol + ((q >> 2) + y) * 32, w);      // (beyond the last atom: zeros into columns of this operand)
                    }
                }
                if (CONVERT) nrm_next = nrm_s[tid];
                tmem_wait_st();
            }
            fence_before();
            bar_arrive(BAR(S::UEMPTY));
            bar_arrive(BAR(S::AFULL + half));
        };
        int dense_next = 0;
        auto ahead = [&](int64_t i) {                        // what the next tile starts with, and is not waited for then
            if (!CONVERT) {
                const int64_t r = (blockIdx.x + i * gridDim.x) * SCR_TILE + tid;
                nrm_next = (i < ntl && r < p.n) ? __ldg(p.n2 + r) : 0.f;
            }
            dense_next = __ldcg(p.ctl + SC_DENSE);
        };
        ahead(0);
        if (ntl > 0) operand(0);
        for (int64_t i = 0; i < ntl; ++i) {
            const int64_t wrow = (blockIdx.x + i * gridDim.x) * SCR_TILE + warp * 32;       // first row of this warp
            const int64_t row = wrow + lane;
            const bool in = row < p.n;
            const float nrm = nrm_next;
            if (__any_sync(0xffffffffu, dense_next != 0)) {  // (some CTA has found the data dense: all roles leave)
                *abort_flag = 1;
                break;
            }
            float thr = -CUDART_INF_F;                       // the largest lower bound so far
            float low[TOP];                                  // TOP > 1: the largest ones, in order
#pragma unroll
            for (int j = 0; j < TOP; ++j) low[j] = -CUDART_INF_F;
            // what a value has to reach
            auto floor_now = [&]() -> float { return TOP == 1 ? thr - p.margin : fmaxf(fminf(low[0] - p.margin, low[TOP - 1]), 0.5f * SCR_NEVER); };
            int ne = 0, packs = 0;
            float lost = -CUDART_INF_F;                      // largest upper bound of a block with marks that found no room
            // The largest of the four quarters of 32 accumulators (= the point's approximate values for a block of components).
            auto quarters = [&](const uint32_t (&v)[32], float (&mx)[4]) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    mx[j] = max3(__uint_as_float(v[8 * j]), __uint_as_float(v[8 * j + 1]), __uint_as_float(v[8 * j + 2]));
                    mx[j] = max3(mx[j], __uint_as_float(v[8 * j + 3]), __uint_as_float(v[8 * j + 4]));
                    mx[j] = max3(mx[j], __uint_as_float(v[8 * j + 5]), __uint_as_float(v[8 * j + 6]));
                }
                if (TOP == 1) {                              // (the quarters themselves are not asked for)
                    mx[0] = max3(mx[0], __uint_as_float(v[7]), __uint_as_float(v[15]));
                    mx[1] = max3(mx[1], __uint_as_float(v[23]), __uint_as_float(v[31]));
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) mx[j] = fmaxf(mx[j], __uint_as_float(v[8 * j + 7]));
                }
            };
            // a block's mask, its largest upper bound rounded up to the 24 bits that share a word with its number
            auto entry = [&](float ub, int bn, unsigned mask) -> unsigned long long {
                return ((unsigned long long)((__float_as_uint(ub + fabsf(ub) * 1e-4f + 1e-3f) & ~255u) | (unsigned)bn) << 32) | mask;
            };
            // marks that found no room in shared memory, or no useful bound
            auto later = [&](int bn, float bmax, float E, unsigned mask) {
                if (!(floor_now() - E > 0.5f * SCR_NEVER)) { // no useful bound (yet): the values of positions without a component could
                    lost = CUDART_INF_F;                     // pass, so the row is evaluated in full
                    return;
                }
                if (ne == S::ENT + S::SPILL && packs < 2) {  // drop what the bound found meanwhile rules out (of broad posteriors:
                    int m = 0;                               // nothing; trying at every block took a millisecond per tile)
                    ++packs;
                    for (int e = 0; e < S::ENT + S::SPILL; ++e) {
                        const unsigned long long o = ent(e);
                        if (__uint_as_float((unsigned)(o >> 32) & ~255u) >= floor_now()) ent(m++) = o;
                    }
                    ne = m;
                }
                if (ne < S::ENT + S::SPILL) ent(ne++) = entry(bmax + E, bn, mask);
                else lost = fmaxf(lost, bmax + E);           // (harmless if the final bound rules the block out)
            };
            // Marks of a block with largest value bmax and allowance E.  CONVERT: the rare cases after the group's four blocks, in one copy
            // of their code (block `at`, its mask in `mask`): the loop over the groups shares the instruction cache with the converting warps
            // (1.02M x 128, K = 1024: 436 us, with a copy per block 450; without those warps 298 and 282 us at D = 64).
            auto mark = [&](const uint32_t (&v)[32], int at, int bn, float bmax, float E, unsigned& mask, unsigned& rest) {
                const float cut = floor_now() - E;
                if (in && bmax >= cut) {
                    // bit j of the mask: value j reaches the cut (the sign of l - cut; four chains of shifts, a byte each)
                    const uint64_t nc = pack2(__float_as_uint(-cut), __float_as_uint(-cut));
                    unsigned m4[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int j = 3; j >= 0; --j)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint64_t d = add2(pack2(v[8 * q + 2 * j], v[8 * q + 2 * j + 1]), nc);
                            m4[q] = __funnelshift_l(__float_as_uint(hi2(d)), m4[q], 1);
                            m4[q] = __funnelshift_l(__float_as_uint(lo2(d)), m4[q], 1);
                        }
                    mask = ~((m4[0] | (m4[1] << 8)) | ((m4[2] << 16) | (m4[3] << 24)));
                    if (cut > 0.5f * SCR_NEVER && ne < S::ENT) ent_s[256 * ne++] = entry(bmax + E, bn, mask);
                    else if (CONVERT) rest |= 1u << at;
                    else later(bn, bmax, E, mask);
                }
            };
            for (int gg = 0; gg < GT; ++gg, ++gi) {
                const bool last = gg + 1 == GT, again = gg == NG;
                const int g = again ? 0 : gg;
                if (last) ahead(i + 1);
                const bool got = bar_wait(BAR(S::LFULL + half), gi & 1u, abort_flag, p.status, false);
                const bool ok = __all_sync(0xffffffffu, got);
                fence_after();
                if (last && i + 1 < ntl) operand(i + 1);     // (the tile's last products are done: its operand is free)
                // the whole group into registers: the tensor cores may overwrite the columns while it is worked through
                uint32_t v0[32], v1[32], v2[32], v3[32];
                tmem_ld32(col, v0);
                tmem_ld32(col + 32, v1);
                tmem_ld32(col + 64, v2);
                tmem_ld32(col + 96, v3);
                tmem_wait(v0); tmem_wait(v1); tmem_wait(v2); tmem_wait(v3);
                fence_before();
                bar_arrive(BAR(S::LEMPTY + half));
                if (ok) {
                    // (the four blocks' maxima first, then their marks: four independent chains, and a bound that has seen the whole
                    // group; block by block the chains of one another kept the warp waiting)
                    float q0[4], q1[4], q2[4], q3[4], bm[4], E[4];
                    quarters(v0, q0); quarters(v1, q1); quarters(v2, q2); quarters(v3, q3);
                    bm[0] = fmaxf(max3(q0[0], q0[1], q0[2]), q0[3]); bm[1] = fmaxf(max3(q1[0], q1[1], q1[2]), q1[3]);
                    bm[2] = fmaxf(max3(q2[0], q2[1], q2[2]), q2[3]); bm[3] = fmaxf(max3(q3[0], q3[1], q3[2]), q3[3]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 ab = blk[4 * g + j];
                        E[j] = fmaf(ab.y, nrm, fabsf(ab.x));
                        if (TOP == 1) {
                            thr = fmaxf(thr, ab.x < 0.f ? -CUDART_INF_F : bm[j] - E[j]);
                        } else if (!again && !(ab.x < 0.f) && bm[j] - E[j] > low[TOP - 1]) {
                            const float (&mx)[4] = j == 0 ? q0 : j == 1 ? q1 : j == 2 ? q2 : q3;
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                float x = mx[q] - E[j];
#pragma unroll
                                for (int t = 0; t < TOP; ++t) {
                                    const float keep = fmaxf(low[t], x);
                                    x = fminf(low[t], x);
                                    low[t] = keep;
                                }
                            }
                        }
                    }
                    if (TOP == 1 || gg > 0) {
                        unsigned mk[4] = {0u, 0u, 0u, 0u}, rest = 0u;
                        mark(v0, 0, 4 * g, bm[0], E[0], mk[0], rest);
                        mark(v1, 1, 4 * g + 1, bm[1], E[1], mk[1], rest);
                        mark(v2, 2, 4 * g + 2, bm[2], E[2], mk[2], rest);
                        mark(v3, 3, 4 * g + 3, bm[3], E[3], mk[3], rest);
#pragma unroll 1
                        while (rest) {
                            const int j = __ffs(rest) - 1;
                            rest &= rest - 1;
                            later(4 * g + j, j == 0 ? bm[0] : j == 1 ? bm[1] : j == 2 ? bm[2] : bm[3], j == 0 ? E[0] : j == 1 ? E[1] : j == 2 ? E[2] : E[3],
                                  j == 0 ? mk[0] : j == 1 ? mk[1] : j == 2 ? mk[2] : mk[3]);
                        }
                    }
                }
            }
            // the point's list: the words (block of 32 positions, mask) that the final bound leaves
            int cnt = 0, nw = 0;
            const float fin = floor_now();
            bool over = !(nrm < CUDART_INF_F) || (lost >= fin && lost > -CUDART_INF_F);
            // (the entries in shared memory all at once: one after the other, each waited for, they took ten times as long,
            // and the tensor cores waited with them)
            unsigned long long we[S::ENT];
            unsigned keep = 0;
#pragma unroll
            for (int e = 0; e < S::ENT; ++e) we[e] = ent_s[256 * e];
#pragma unroll
            for (int e = 0; e < S::ENT; ++e)
                if (e < ne && __uint_as_float((unsigned)(we[e] >> 32) & ~255u) >= fin) {
                    cnt += __popc((unsigned)we[e]);
                    keep |= 1u << e;
                }
            for (int e = S::ENT; e < ne; ++e) {
                const unsigned long long w = ent(e);
                if (__uint_as_float((unsigned)(w >> 32) & ~255u) >= fin) {
                    cnt += __popc((unsigned)w);
                    keep |= 1u << e;
                }
            }
            if (!in || over) cnt = 0, keep = 0;
            nw = __popc(keep);
            if (cnt < TOP || nw > 15) over = true;                      // (a point further from everything than a float16 sum can tell)
            if (over) cnt = nw = 0, keep = 0;
            int inc = cnt | (nw << 16);                      // running sums of both over the warp
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if ((inc & 0xffff) > 32 * SCR_SLOTS || (inc >> 16) > 32 * SCR_WORDS) over = true;
            if (in && !*abort_flag) {
                const int wo = (inc >> 16) - nw;
                p.pt_off[row] = (unsigned)(wrow * SCR_SLOTS) + (unsigned)((inc & 0xffff) - cnt);
                p.pt_cnt[row] = (over || cnt == 0) ? 0 : (wo << 16) | (nw << 12) | cnt;
                if (over) {
                    p.ovf[atomicAdd(p.ctl + SC_OVF, 1)] = (int)row;
                } else {
                    marks += cnt;
                    uint2* o = p.words + wrow * SCR_WORDS + wo;
#pragma unroll
                    for (int e = 0; e < S::ENT; ++e)
                        if (keep >> e & 1u) *o++ = make_uint2((unsigned)we[e], (unsigned)(we[e] >> 32) & 255u);
                    for (int e = S::ENT; e < ne; ++e)
                        if (keep >> e & 1u) {
                            const unsigned long long w = ent(e);
                            *o++ = make_uint2((unsigned)w, (unsigned)(w >> 32) & 255u);
                        }
                }
            }
        }
        if (ntl > 0 && !*abort_flag) {
            marks = __reduce_add_sync(0xffffffffu, marks);
            if (lane == 0 && marks > 0) atomicAdd(p.ctl + SC_MARKS, marks);
        }
    } else if (CONVERT && warp < S::PRODUCER) {
        // =========================== converting warps: rows of X -> rows of u, |u|^2 ===========================
        give_registers();
        switch (screen_lane_shift(p.KC)) {
            case 1: screen_convert<1>(p, smem, warp - S::CONVERTER, lane, (int)ntl, abort_flag); break;
            case 2: screen_convert<2>(p, smem, warp - S::CONVERTER, lane, (int)ntl, abort_flag); break;
            case 3: screen_convert<3>(p, smem, warp - S::CONVERTER, lane, (int)ntl, abort_flag); break;
            default: screen_convert<4>(p, smem, warp - S::CONVERTER, lane, (int)ntl, abort_flag); break;
        }
    } else if (give_registers(), role == S::PRODUCER) {
        // =========================== producer warp (bulk copies of the coefficients) ===========================
        uint32_t ps = 0, slot = 0, phase = 1, cslot = 0;     // stages requested so far; the next one's slot and its phase; slot of the group's constants
        bool ok = true;
        auto wait_slot = [&](int bar, uint32_t parity) -> bool {
            uint32_t w = 1;
            if (lane == 0) w = bar_wait(BAR(bar), parity, abort_flag, p.status, false) ? 1u : 0u;
            return __shfl_sync(0xffffffffu, w, 0) != 0u;
        };
        auto bulk = [&](unsigned char* dst, const unsigned char* src, uint32_t bytes, uint32_t bar) {
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(bar) : "memory");
        };
        uint32_t ut = 0;                                     // tiles whose rows have been requested
        const uint32_t ubytes = 256u * 16u * (uint32_t)p.chunks;
        auto load_rows = [&](int64_t i) {
            if (elect_one()) {
                const unsigned char* src = p.y + (size_t)((blockIdx.x + i * gridDim.x) * SCR_TILE) * p.chunks * 16;
                bar_expect_tx(BAR(S::UFULL), ubytes);
                bulk(smem + S::UOFF, src, ubytes, BAR(S::UFULL));
            }
            __syncwarp();
            ++ut;
        };
        if (!CONVERT && ntl > 0) load_rows(0);
        for (int64_t i = 0; i < ntl && ok; ++i)
            for (int g = 0; g < GT && ok; ++g) {
                for (int z = 0; z < spg && ok; ++z) {
                    if (ps >= S::PS) ok = wait_slot(S::PEMPTY + slot, phase);
                    if (!ok) break;
                    if (elect_one()) {
                        const unsigned char* src = p.img + (size_t)(g == NG ? 0 : g) * p.gbytes;
                        const uint32_t bytes = min(p.KA - 2 * z, 2) * 16384u;
                        bar_expect_tx(BAR(S::PFULL + slot), bytes + (z == 0 ? SW_CSLOT : 0));
                        if (z == 0) bulk(cons + cslot * SW_CSLOT, src, SW_CSLOT, BAR(S::PFULL + slot));
                        bulk(smem + slot * SW_PSLOT, src + SW_CSLOT + z * SW_PSLOT, bytes, BAR(S::PFULL + slot));
                    }
                    __syncwarp();
                    ++ps;
                    if (++slot == S::PS) { slot = 0; phase ^= 1u; }
                }
                if (++cslot == (uint32_t)S::CSLOTS) cslot = 0;
                // the next tile's rows as soon as both halves have taken this tile's (which they do before its first products);
                // no stage waits for that except behind the tile's last one
                if (!CONVERT && ok && ut == (uint32_t)(i + 1) && i + 1 < ntl) {
                    uint32_t free_now = (g + 1 == GT) ? 1u : 0u;
                    if (free_now) ok = wait_slot(S::UEMPTY, (uint32_t)(i & 1));
                    else {
                        if (lane == 0) free_now = bar_test(BAR(S::UEMPTY), (uint32_t)(i & 1)) ? 1u : 0u;
                        free_now = __shfl_sync(0xffffffffu, free_now, 0);
                    }
                    if (ok && free_now) load_rows(i + 1);
                }
            }
        // the loads in flight must have landed before the CTA may exit, also where the others leave after the last one has been asked for
        for (uint32_t h = (ps > S::PS ? ps - S::PS : 0); h < ps; ++h) {
            if (lane == 0) bar_wait(BAR(S::PFULL + h % S::PS), (h / S::PS) & 1u, drain_flag, p.status, false);
            __syncwarp();
        }
        if (!CONVERT && ut > 0 && lane == 0) bar_wait(BAR(S::UFULL), (ut - 1) & 1u, drain_flag, p.status, false);
        __syncwarp();
    } else if (CONVERT && role == S::FETCH) {
        // =========================== the warp that fetches X ===========================
        const SweepRows rows(p, screen_lane_shift(p.KC));
        const int total = (int)ntl * rows.per;
        int c = 0;
        bool ok = true;
        for (int i = 0; i < (int)ntl && ok; ++i)
            for (int k = 0; k < rows.per; ++k, ++c) {
                const uint32_t full = BAR(S::XFULL + (c & 1));
                if (c >= 2) {
                    uint32_t w = 1;
                    if (lane == 0) w = bar_wait(BAR(S::XEMPTY + (c & 1)), (uint32_t)((c >> 1) - 1) & 1u, abort_flag, p.status, false) ? 1u : 0u;
                    ok = __shfl_sync(0xffffffffu, w, 0) != 0u;
                    if (!ok) break;
                }
                const int row0 = rows.first + i * rows.tstep + k * rows.R;
                uint32_t lo, bytes;
                const bool bulk = rows.range(row0, lo, bytes);
                if (elect_one()) {
                    if (bulk) {
                        bar_expect_tx(full, bytes);
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     ::"r"(smem_u32(smem + S::XOFF + (c & 1) * SW_XBYTES)), "l"(rows.xb + lo), "r"(bytes), "r"(full) : "memory");
                    } else {
                        bar_arrive(full);
                    }
                    // two chunks alone do not cover the trip to memory: the one after them is on its way into L2
                    const int ahead = c + 2 >= total ? -1 : k + 2 < rows.per ? row0 + 2 * rows.R : row0 + 2 * rows.R + (k + 2) / rows.per * (rows.tstep - SCR_TILE);
                    if (ahead >= 0 && rows.range(ahead, lo, bytes))
                        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(rows.xb + lo), "r"(bytes) : "memory");
                }
                __syncwarp();
            }
        // the copies in flight must have landed before the CTA may exit, also after an abort
        for (int q = c > 2 ? c - 2 : 0; q < c; ++q) {
            if (lane == 0) bar_wait(BAR(S::XFULL + (q & 1)), (uint32_t)(q >> 1) & 1u, drain_flag, p.status, false);
            __syncwarp();
        }
    } else {
        // =========================== MMA warps, one per half ===========================
        // An instruction takes about as long to issue as the tensor cores take for it, and few are queued: every cycle spent
        // between two of them is idle time of the tensor cores unless the other half's warp fills it.  So there is a warp per
        // half, one thread of it does all (no votes, no shuffles), and a stage is waited for only when the instructions of the
        // stage before it have been issued.
        const int h = role - S::MMA;
        if (elect_one()) {
            const uint32_t idesc = make_idesc(128, 128, 0);
            const uint64_t dp = make_desc(smem_u32(smem), 16, 1024);
            const uint64_t dc = make_desc32(smem_u32(cons)), da = make_desc32(smem_u32(smem + S::AOFF));
            const uint32_t d = tmem + h * 128, a = tmem + 256 + h * 128;
            const uint32_t bars0 = BAR(0);
            auto wait = [&](int bar, uint32_t parity) -> bool { return bar_wait(bars0 + 8 * bar, parity, abort_flag, p.status, false); };
            uint32_t slot = 0, parity = 0, cslot = 0;        // of the next stage; of the group's constants
            uint32_t gi = 0;
            bool alive = true;
            for (int64_t i = 0; i < ntl && alive; ++i) {
                for (int g = 0; g < GT && alive; ++g, ++gi) {
                    if (g == 0) alive = wait(S::AFULL + h, (uint32_t)(i & 1));
                    if (alive && gi >= 1) alive = wait(S::LEMPTY + h, (gi - 1) & 1u);
                    for (int z = 0; z < spg && alive; ++z) {
                        if (!wait(S::PFULL + slot, parity)) { alive = false; break; }
                        fence_after();
                        if (z == 0) mma_ss(d, da, dc + ((cslot * SW_CSLOT) >> 4), idesc, 0u);      // the constants
                        const int nk = p.KS - 8 * z;         // k-steps of this stage: at most eight
                        const uint64_t b = dp + ((slot * SW_PSLOT) >> 4);
                        if (nk >= 8) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) mma_ts(d, a + z * 64 + j * 8, b + (((j >> 2) * 16384 + (j & 3) * 32) >> 4), idesc, 1u);
                        } else {
#pragma unroll
                            for (int j = 0; j < 7; ++j)
                                if (j < nk) mma_ts(d, a + z * 64 + j * 8, b + (((j >> 2) * 16384 + (j & 3) * 32) >> 4), idesc, 1u);
                        }
                        mma_commit(bars0 + 8 * (S::PEMPTY + slot));
                        if (++slot == S::PS) { slot = 0; parity ^= 1u; }
                    }
                    if (alive && !(p.test_silent == (int)blockIdx.x && gi == 0)) mma_commit(bars0 + 8 * (S::LFULL + h));
                    if (++cslot == (uint32_t)S::CSLOTS) cslot = 0;
                }
            }
            mma_commit(bars0 + 8 * (S::FINAL + h));
            bar_wait(bars0 + 8 * (S::FINAL + h), 0, drain_flag, p.status, false);
            fence_after();
        }
        __syncwarp();
    }
    fence_before();
    __syncthreads();
    // A CTA that left early has not written its points' lists, and what was in that memory before must not be taken for offsets and
    // components: nothing after this kernel does anything, also when a wait ran out.
    if (threadIdx.x == 0 && (abort_s != 0 || drain_s != 0)) p.ctl[SC_DENSE] = 1;
    if (warp == S::MMA) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_maxf(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Rows that left the sweep without a list (marks in too many groups of components, a coordinate beyond the fp16 range): all K
// components exactly, the list from those values.  Four rows per CTA and step, a warp per component.  Also the verdict on the
// piece: with too many such rows, or too many pairs, SC_DENSE is set and nothing after this kernel does anything.
constexpr int OV_ROWS = 4;
__global__ void __launch_bounds__(256) screen_rows_kernel(const float* __restrict__ X, int64_t n, int D, int K, float margin, int top,
                                                          long long max_marks, const float* __restrict__ mu, const float* __restrict__ w2,
                                                          const double* __restrict__ c2d, const int* __restrict__ ovf,
                                                          unsigned* __restrict__ pt_off, int* __restrict__ pt_cnt,
                                                          unsigned short* __restrict__ ids, int* __restrict__ ctl) {
    if (screen_off(ctl)) return;
    const int rows = ctl[SC_OVF];
    if ((long long)rows * 32 > n + 1024 || (long long)ctl[SC_MARKS] > max_marks) {
        if (threadIdx.x == 0) ctl[SC_DENSE] = 1;     // (any number of CTAs may write the same value)
        return;
    }
    extern __shared__ float l_s[];                   // [OV_ROWS][K]
    __shared__ float x_s[OV_ROWS][128];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int r0 = blockIdx.x * OV_ROWS; r0 < rows; r0 += gridDim.x * OV_ROWS) {
        __syncthreads();
        for (int e = tid; e < OV_ROWS * 128; e += 256) {
            const int r = e >> 7, d = e & 127;
            x_s[r][d] = (r0 + r < rows && d < D) ? __ldg(X + (int64_t)ovf[r0 + r] * D + d) : 0.f;
        }
        __syncthreads();
        for (int k = warp; k < K; k += 8) {
            float q[OV_ROWS] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int d = lane + 32 * i;
                if (d >= D) continue;
                const float m = __ldg(mu + (size_t)k * D + d), w = __ldg(w2 + (size_t)k * D + d);
#pragma unroll
                for (int r = 0; r < OV_ROWS; ++r) { const float t = x_s[r][d] - m; q[r] = fmaf(w * t, t, q[r]); }
            }
#pragma unroll
            for (int r = 0; r < OV_ROWS; ++r) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) q[r] += __shfl_xor_sync(0xffffffffu, q[r], o);
            }
            const float c = (float)__ldg(c2d + k);
            if (lane < OV_ROWS) l_s[(size_t)lane * K + k] = c - (lane == 0 ? q[0] : lane == 1 ? q[1] : lane == 2 ? q[2] : q[3]);
        }
        __syncthreads();
        if (warp < OV_ROWS && r0 + warp < rows) {
            const float* l = l_s + (size_t)warp * K;
            float best = -CUDART_INF_F;
            for (int k = lane; k < K; k += 32) best = fmaxf(best, l[k]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
            float cut = best - margin - 0.01f;
            if (top > 1) {                                   // and what the `top` largest reach (-inf: all components)
                float kth = CUDART_INF_F;
                for (int left = top; left > 0;) {
                    float b = -CUDART_INF_F;
                    int same = 0;
                    for (int k = lane; k < K; k += 32) {
                        const float v = l[k];
                        if (v < kth) { if (v > b) { b = v; same = 1; } else if (v == b) ++same; }
                    }
                    const float m = warp_maxf(b);
                    left -= __reduce_add_sync(0xffffffffu, b == m ? same : 0);
                    kth = m;
                    if (m == -CUDART_INF_F) break;
                }
                cut = fminf(cut, kth);
            }
            int cnt = 0;
            for (int k0 = 0; k0 < K; k0 += 32) {
                const bool is = k0 + lane < K && best > -CUDART_INF_F && l[k0 + lane] >= cut;
                cnt += __popc(__ballot_sync(0xffffffffu, is));
            }
            int base = 0;
            if (lane == 0) base = atomicAdd(ctl + SC_EXTRA, cnt);
            base = __shfl_sync(0xffffffffu, base, 0);
            const bool fits = (long long)base + cnt <= (long long)SCR_PIECE * SCR_EXTRA;
            const unsigned o = (unsigned)(SCR_PIECE * SCR_SLOTS) + (unsigned)base;
            const int row = ovf[r0 + warp];
            if (lane == 0) {
                if (!fits) ctl[SC_DENSE] = 1;
                pt_off[row] = fits ? o : 0;
                pt_cnt[row] = fits ? cnt : 0;
            }
            int done = 0;
            for (int k0 = 0; fits && k0 < K; k0 += 32) {
                const bool is = k0 + lane < K && best > -CUDART_INF_F && l[k0 + lane] >= cut;
                const unsigned b = __ballot_sync(0xffffffffu, is);
                if (is) ids[o + done + __popc(b & ((1u << lane) - 1u))] = (unsigned short)(k0 + lane);
                done += __popc(b);
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Exact values.  A CTA takes a range of consecutive points, a third of an SM each, all of a piece in one wave.  Points with one mark alone need no
// value (of a step) and are done first.  The others are put in order of their first mark (`sorted`), so that points of one cluster,
// whose marks are much the same, come together and the components' rows (1 KB per pair at D = 128) out of L1.  Then a warp takes 32 points
// at a time, their marks as lists in shared memory, and four of them at once, eight lanes each: the point's row in registers, a lane with every eighth
// group of four dimensions, the pairs' sums added up eight at a time, so that a step waits for nothing but its rows.
// Bound by the trips of a step to L1 and L2 (1200 cycles with 24 warps on an SM) and their wavefronts.  1.2M x 100, K = 1000 (2.4 marks per point): 334 us with
// four pairs of 32 consecutive points per step, each of which fetched the point's row and the component's rows, mostly from L2, and had its three shuffles
// and its constant at its end; 231 now.  Not kept: rows of the next pair in flight (registers: two CTAs per SM), four rows of the first part per lane
// (spills), prefetches of the points' rows into L2 (no gain).
constexpr int EV_VALS = 32 * SCR_SLOTS;
constexpr int EV_KEYS = 1024;                // keys of the sort (positions in the sweep, neighbours together beyond so many)
constexpr int EV_RANGE = (int)((SCR_PIECE + SCR_RANGES - 1) / SCR_RANGES + 31) / 32 * 32;      // most points of a CTA
constexpr int EV_BATCHES = EV_RANGE / 32 + 8;
// TOP: the m (<= 4) largest values go out, the smaller component first where two are equal.
struct TopOut { int m; float* resp; ScreenTie tie; };

// Two centroids at the same distance but for rounding: one such point in a small cluster moves its centroid, so the nearest-centroid
// search decides near ties in the arithmetic of the kernels that take the call when the posteriors are broad.  The whole warp, one
// point: all its candidates within `near` of the best.
__device__ int screen_nearest(const ScreenTie& tie, const float* __restrict__ x, int D, const float* __restrict__ mu, const float* l_s,
                              const unsigned short* k_s, int cnt, float mx, float near, int lane) {
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(x) & 15) == 0);
    float bv = -CUDART_INF_F;
    int bk = 0x7fffffff;
    for (int j = 0; j < cnt; ++j) {
        if (!(l_s[j] >= mx - near)) continue;                // warp-uniform
        const int k = k_s[j];
        const float* m = mu + (size_t)k * D;
        float q = 0.f;
        if (tie.g == nullptr) {                              // as the refinement of the tensor assignment: 4 dimensions per lane, butterfly
            for (int t = 0; t < 4; ++t) {
                const int d = vec ? 4 * lane + t : lane + 32 * t;
                if (d < D) { const float diff = __ldg(x + d) - __ldg(m + d); q = fmaf(diff * diff, tie.w, q); }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        } else {                                             // as the FP32 tile kernel: one chain about the centre
            for (int d = 0; d < D; ++d) {
                const float g = __ldg(tie.g + d), t = fmaf(__ldg(x + d) - g, 1.f, g - __ldg(m + d));
                q = fmaf(t, t, q);
            }
        }
        const float e = tie.c - q;
        if (e > bv || (e == bv && k < bk)) { bv = e; bk = k; }
    }
    return bk;
}

template <int MODE, int NX, bool VEC>
__global__ void __launch_bounds__(256, 3) screen_eval_kernel(const float* __restrict__ X, int64_t n, int D, int K, const float* __restrict__ mu,
                                                             const float* __restrict__ w2, const double* __restrict__ c2d,
                                                             const int* __restrict__ comp_of, int range, int sorted,
                                                             const uint2* __restrict__ words,
                                                             const unsigned* __restrict__ pt_off, int* __restrict__ pt_cnt,
                                                             unsigned short* __restrict__ ids, float* __restrict__ val,
                                                             int* __restrict__ counts, double* __restrict__ ll, float* __restrict__ logp,
                                                             int32_t* __restrict__ idx, int* __restrict__ ctl, const TopOut top) {
    if (ctl[SC_DENSE] != 0) return;
    if (blockIdx.x == 0 && threadIdx.x < 3) ctl[SC_MARKS + threadIdx.x] = 0;       // (for the next piece's sweep)
    // (a piece is done with its last kernel: this one where there are no statistics)
    if ((MODE == SCREEN_LOGP || MODE == SCREEN_TOP) && blockIdx.x == 0 && threadIdx.x == 0) ctl[SC_DONE] += 1;
    extern __shared__ int hist[];                    // [K] (unless MODE == SCREEN_LOGP or SCREEN_TOP), `keys`, `order`
    __shared__ __align__(16) unsigned char work_s[8 * EV_VALS * 6];
    __shared__ uint4 pt_s[8][32];                    // the points of a batch: row, where its pairs start here and in the lists, how many there are
    __shared__ double ll_s[EV_BATCHES];              // log-likelihoods of the batches (a warp takes the next one when it is done with one)
    __shared__ double red_s[8];
    __shared__ int wsum[8];
    __shared__ int next_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l8 = lane & 7, grp = lane >> 3;
    float* const v_s = reinterpret_cast<float*>(work_s) + warp * EV_VALS;          // values of the warp's pairs
    unsigned short* const k_s = reinterpret_cast<unsigned short*>(work_s + 8 * EV_VALS * 4) + warp * EV_VALS;       // their positions in the sweep, then their components
    unsigned* const cur32 = reinterpret_cast<unsigned*>(work_s);                   // (while the points are sorted) [8][EV_KEYS] 16-bit cursors
    const bool histogram = MODE != SCREEN_LOGP && MODE != SCREEN_TOP && counts != nullptr;
    short* const keys = reinterpret_cast<short*>(hist + (MODE != SCREEN_LOGP && MODE != SCREEN_TOP ? K : 0));       // [range] of the points of the last part; else -1
    unsigned short* const order = reinterpret_cast<unsigned short*>(keys + range);                                  // [range] the points of the last part
    if (histogram)
        for (int k = tid; k < K; k += 256) hist[k] = 0;
    if (sorted)
        for (int k = tid; k < 4 * EV_KEYS; k += 256) cur32[k] = 0u;
    if (tid == 0) next_s = 0;
    if (lane == 0) wsum[warp] = 0;
    __syncthreads();
    // A row (of X or of the parameters), NX x 4 values of it in each of the eight lanes that work on a point: dimensions 4 (l8 + 8 i) + (0..3), or, where rows
    // cannot be read 16 bytes at a time, l8 + 8 (4 i + (0..3)).  Beyond D zeros.
    auto row_of = [&](const float* __restrict__ r, uint64_t (&v)[2 * NX]) {
#pragma unroll
        for (int i = 0; i < NX; ++i) {
            if constexpr (VEC) {
                ulonglong2 a = make_ulonglong2(0ull, 0ull);
                if (i < NX - 1 || 4 * (l8 + 8 * i) < D) a = __ldg(reinterpret_cast<const ulonglong2*>(r) + l8 + 8 * i);
                v[2 * i] = a.x;
                v[2 * i + 1] = a.y;
            } else {
                float f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) f[j] = i < NX - 1 || l8 + 8 * (4 * i + j) < D ? __ldg(r + l8 + 8 * (4 * i + j)) : 0.f;
                v[2 * i] = pack2(__float_as_uint(f[0]), __float_as_uint(f[1]));
                v[2 * i + 1] = pack2(__float_as_uint(f[2]), __float_as_uint(f[3]));
            }
        }
    };
    // This lane's part of sum_d w (x - m)^2.
    auto part_of = [&](const uint64_t (&xv)[2 * NX], int k) -> float {
        uint64_t m[2 * NX], w[2 * NX], q2 = 0ull;
        row_of(mu + (size_t)k * D, m);
        row_of(w2 + (size_t)k * D, w);
#pragma unroll
        for (int i = 0; i < 2 * NX; ++i) {
            const uint64_t t = sub2(xv[i], m[i]);
            q2 = fma2(mul2(w[i], t), t, q2);
        }
        return lo2(q2) + hi2(q2);
    };
    auto value_of = [&](int k, float q) -> float { return (float)(__ldg(c2d + k) - (double)q); };
    double ll_acc = 0.0;
    const int64_t first = (int64_t)blockIdx.x * range;
    const int rows = (int)((n - first < range) ? n - first : range);
    // A point's list: where its words are, and how many marks they hold (off beyond the lists of the sweep: a list of its own length).
    struct List { unsigned off; int cnt, nw; bool listed; };
    auto list_of = [&](int64_t row, int pc) -> List {
        List a;
        a.off = pt_off[row];
        a.listed = a.off < (unsigned)(SCR_PIECE * SCR_SLOTS);
        a.cnt = a.listed ? pc & 4095 : pc;
        a.nw = a.listed ? (pc >> 12) & 15 : 0;
        return a;
    };
    auto words_of = [&](int64_t row, int pc) { return words + (row & ~(int64_t)31) * SCR_WORDS + (pc >> 16); };      // (32 points of the sweep share a part of the lists)
    auto first_of = [&](const uint2* w) { const uint2 a = __ldg(w); return (int)a.y * 32 + __ffs(a.x) - 1; };
    const int key_shift = K <= EV_KEYS ? 0 : 32 - __clz((K - 1) / EV_KEYS);        // (positions: below K rounded up to 128)

    // ---- points whose values are not needed here, and rows with lists of their own length
    for (int r0 = warp * 32; r0 < rows; r0 += 256) {
        const int64_t row0 = first + r0, row = row0 + lane;
        const bool in = r0 + lane < rows;
        const int pc = in ? pt_cnt[row] : 0;
        List a = {0u, 0, 0, true};
        if (in) a = list_of(row, pc);
        const bool alone = a.listed && a.cnt == 1 && MODE != SCREEN_LOGP, lone_list = a.cnt > 0 && !a.listed;
        const bool todo = a.listed && a.cnt > 0 && !alone;
        const unsigned todos = __ballot_sync(0xffffffffu, todo);
        int mark = 0;
        if (alone || (sorted && todo)) mark = first_of(words_of(row, pc));
        const int key = todo ? min(mark >> key_shift, EV_KEYS - 1) : -1;
        if (r0 + lane < range) keys[r0 + lane] = (short)key;
        if (sorted) { if (todo) atomicAdd(cur32 + (warp * EV_KEYS + key) / 2, 1u << (16 * (key & 1))); }
        else if (lane == 0) wsum[warp] += __popc(todos);
        const int only = alone ? __ldg(comp_of + mark) : 0;
        float mx = -CUDART_INF_F, sum = 0.f;
        int best = only, kept = 0;
        // the whole warp, one row after the other, values in `val`
        for (unsigned todo_rows = __ballot_sync(0xffffffffu, lone_list); todo_rows;) {
            const int src = __ffs(todo_rows) - 1;
            todo_rows &= todo_rows - 1;
            const int c = __shfl_sync(0xffffffffu, a.cnt, src);
            const unsigned o = __shfl_sync(0xffffffffu, a.off, src);
            float m = -CUDART_INF_F, sm = 0.f;
            int b = 0;
            uint64_t xv[2 * NX];
            row_of(X + (row0 + src) * D, xv);
            for (int s = 0; s < c; s += 4) {
                const int j = min(s + (lane >> 3), c - 1);
                const int k = ids[o + j];
                float q = part_of(xv, k);
                q += __shfl_xor_sync(0xffffffffu, q, 1);
                q += __shfl_xor_sync(0xffffffffu, q, 2);
                q += __shfl_xor_sync(0xffffffffu, q, 4);
                const float l = value_of(k, q);
                if (l8 == 0 && s + (lane >> 3) < c) {
                    val[o + j] = l;
                    if (MODE == SCREEN_ARGMAX) { if (l > m || (l == m && k < b)) { m = l; b = k; } }
                    else m = fmaxf(m, l);
                }
            }
#pragma unroll
            for (int x = 16; x > 0; x >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, m, x);
                const int ob = __shfl_xor_sync(0xffffffffu, b, x);
                if (om > m || (om == m && ob < b)) { m = om; b = ob; }
            }
            __syncwarp();
            if (MODE != SCREEN_ARGMAX)
                for (int j = lane; j < c; j += 32) sm += fast_ex2(val[o + j] - m);
#pragma unroll
            for (int x = 16; x > 0; x >>= 1) sm += __shfl_xor_sync(0xffffffffu, sm, x);
            const float ls = log2f(sm), lz = m + ls;
            if (MODE == SCREEN_TOP) {
                float pv = CUDART_INF_F;                     // the pair that went out last
                int pk = -1;
                for (int r = 0; r < top.m; ++r) {
                    float bv = -CUDART_INF_F;
                    int bk = 0x7fffffff;
                    for (int j = lane; j < c; j += 32) {
                        const float v = val[o + j];
                        const int k = ids[o + j];
                        const bool after = v < pv || (v == pv && k > pk);
                        if (after && (v > bv || (v == bv && k < bk))) { bv = v; bk = k; }
                    }
#pragma unroll
                    for (int x = 16; x > 0; x >>= 1) {
                        const float ov = __shfl_xor_sync(0xffffffffu, bv, x);
                        const int ok = __shfl_xor_sync(0xffffffffu, bk, x);
                        if (ov > bv || (ov == bv && ok < bk)) { bv = ov; bk = ok; }
                    }
                    if (lane == 0) {
                        idx[(row0 + src) * top.m + r] = bk == 0x7fffffff ? 0 : bk;
                        if (top.resp) top.resp[(row0 + src) * top.m + r] = fast_ex2(bv - lz);
                    }
                    pv = bv;
                    pk = bk;
                }
            }
            int kp = 0;
            if (MODE == SCREEN_EM)
                for (int j0 = 0; j0 < c; j0 += 32) {
                    const int j = j0 + lane;
                    const float v = j < c ? val[o + j] : -CUDART_INF_F, r = fast_ex2((v - m) - ls);
                    const int id = j < c ? ids[o + j] : 0;
                    const bool keep = r >= 9.094947e-13f;
                    const unsigned bal = __ballot_sync(0xffffffffu, keep);
                    __syncwarp();
                    if (keep) {
                        const int q = kp + __popc(bal & ((1u << lane) - 1u));
                        ids[o + q] = (unsigned short)id;
                        val[o + q] = r;
                        if (histogram) atomicAdd(&hist[id], 1);
                    }
                    kp += __popc(bal);
                    __syncwarp();
                }
            if (lane == src) { mx = m; sum = sm; best = b; kept = kp; }
        }
        if (!in || todo) continue;
        if (MODE == SCREEN_TOP) {
            if (!lone_list)
                for (int r = 0; r < top.m; ++r) {
                    idx[row * top.m + r] = only;
                    if (top.resp) top.resp[row * top.m + r] = alone ? 1.f : CUDART_NAN_F;       // (not a number: no component has a weight)
                }
        } else if (MODE == SCREEN_LOGP) {
            const double lz = a.cnt > 0 ? (double)mx + (double)log2f(sum) : -CUDART_INF;
            logp[row] = (float)(lz * 0.69314718055994530942);
            ll_acc += lz;
        } else if (MODE == SCREEN_ARGMAX) {
            if (idx) idx[row] = best;
            if (histogram && a.cnt > 0) {
                ids[a.off] = (unsigned short)best;
                val[a.off] = -1.f;
                pt_cnt[row] = 1;
                atomicAdd(&hist[best], 1);
            }
        } else if (a.cnt == 0) {
            ll_acc += -CUDART_INF;
        } else if (alone) {
            ids[a.off] = (unsigned short)only;
            val[a.off] = -1.f;
            pt_cnt[row] = 1;
            if (histogram) atomicAdd(&hist[only], 1);
        } else {
            ll_acc += (double)mx + (double)log2f(sum);       // (a list of its own length)
            pt_cnt[row] = kept;
        }
    }
    __syncthreads();

    // ---- the others: by their first mark, or as they come
    int work = 0;                                    // points of the last part
    unsigned short* const cur = reinterpret_cast<unsigned short*>(cur32);
    if (sorted) {
        static_assert(EV_KEYS == 4 * 256, "four keys per thread");
        int c4[4], own = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            c4[j] = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const int v = cur[w * EV_KEYS + 4 * tid + j];
                cur[w * EV_KEYS + 4 * tid + j] = (unsigned short)c4[j];
                c4[j] += v;
            }
            own += c4[j];
        }
        int inc = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        int at = inc - own;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += wsum[w];
            work += wsum[w];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int w = 0; w < 8; ++w) cur[w * EV_KEYS + 4 * tid + j] += (unsigned short)at;
            at += c4[j];
        }
        __syncthreads();
        for (int r0 = warp * 32; r0 < rows; r0 += 256) {
            const int key = r0 + lane < rows ? (int)keys[r0 + lane] : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, key);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            int c = 0;
            if (key >= 0) c = cur[warp * EV_KEYS + key];
            __syncwarp();
            if (key >= 0) {
                if (rank == 0) cur[warp * EV_KEYS + key] = (unsigned short)(c + __popc(peers));
                order[c + rank] = (unsigned short)(r0 + lane);
            }
            __syncwarp();
        }
    } else {
        int at = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += wsum[w];
            work += wsum[w];
        }
        for (int r0 = warp * 32; r0 < rows; r0 += 256) {
            const bool todo = r0 + lane < rows && keys[r0 + lane] >= 0;
            const unsigned todos = __ballot_sync(0xffffffffu, todo);
            if (todo) order[at + __popc(todos & ((1u << lane) - 1u))] = (unsigned short)(r0 + lane);
            at += __popc(todos);
        }
    }
    __syncthreads();
    const int pw = min(32, max(4, (work + 31) / 32 * 4));    // points of a batch: whole rounds of four, something for every warp

    // ---- values
    ll_acc = warp_sum(ll_acc);
    if (lane == 0) red_s[warp] = ll_acc;
    const int batches = (work + pw - 1) / pw;
    for (;;) {
        int bt = 0;
        if (lane == 0) bt = atomicAdd(&next_s, 1);
        bt = __shfl_sync(0xffffffffu, bt, 0);
        if (bt >= batches) break;
        const int j0 = bt * pw;
        const bool in = lane < pw && j0 + lane < work;
        const int at_row = in ? (int)order[j0 + lane] : 0;
        const int64_t row = first + at_row;
        const int pc = in ? pt_cnt[row] : 0;
        List a = {0u, 0, 0, true};
        if (in) a = list_of(row, pc);
        int todo = a.cnt;
        ll_acc = 0.0;
        // (all of them unless points of several parts of the lists have more than EV_VALS pairs together)
        while (__any_sync(0xffffffffu, todo > 0)) {
            int inc = todo;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            const int left = inc > EV_VALS ? todo : 0;
            const int now = todo - left, total = (int)__reduce_max_sync(0xffffffffu, (unsigned)(now > 0 ? inc : 0)), p0 = inc - todo;
            todo = left;
            // the points in order of the number of their pairs (four of them are worked on at a time, as long as the longest list takes)
            int rank = 0, points = 0;
            const int cls = min(now, 8);
#pragma unroll
            for (int c = 8; c > 0; --c) {
                const unsigned is = __ballot_sync(0xffffffffu, cls == c);
                if (cls == c) rank = points + __popc(is & ((1u << lane) - 1u));
                points += __popc(is);
            }
            if (now > 0) {   // the marks one by one
                pt_s[warp][rank] = make_uint4((unsigned)at_row, (unsigned)p0, a.off, (unsigned)now);
                const uint2* wd = words_of(row, pc);
                int at = p0;
                for (int e = 0; e < a.nw; ++e) {
                    uint2 w = __ldg(wd + e);
                    while (w.x) {
                        k_s[at++] = (unsigned short)((int)w.y * 32 + __ffs(w.x) - 1);
                        w.x &= w.x - 1;
                    }
                }
            }
            __syncwarp();
            for (int j = lane; j < total; j += 32) k_s[j] = (unsigned short)__ldg(comp_of + k_s[j]);
            __syncwarp();
            for (int r0 = 0; r0 < points; r0 += 4) {
                const bool have = r0 + grp < points;
                const uint4 pt = pt_s[warp][min(r0 + grp, points - 1)];
                const int64_t prow = first + (int)pt.x;
                const int cnt = have ? (int)pt.w : 0, steps = (int)__reduce_max_sync(0xffffffffu, (unsigned)cnt);
                const unsigned off = pt.z;
                float* const pv = v_s + pt.y;
                unsigned short* const pk = k_s + pt.y;
                uint64_t xv[2 * NX];
                row_of(X + prow * D, xv);
                // eight pairs' parts, then the sums: lane l8 gets that of pair j0 + l8.  (dv: what its value lost in 32 bits, beyond the first eight pairs
                // in the point's part of val.  All points of a component lose alike, as its constant lies between two floats, so it does not average out.)
                float dv = 0.f;
                for (int j0 = 0; j0 < steps; j0 += 8) {
                    float q[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        q[j] = 0.f;
                        if (j0 + j < steps) q[j] = part_of(xv, pk[min(j0 + j, (int)pt.w - 1)]);
                    }
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                        for (int j = 0; j < o; ++j) {
                            const float give = (l8 & o) ? q[j] : q[j + o], keep = (l8 & o) ? q[j + o] : q[j];
                            q[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                        }
                    if (j0 + l8 < cnt) {
                        const double v = __ldg(c2d + pk[j0 + l8]) - (double)q[0];
                        pv[j0 + l8] = (float)v;
                        if (MODE == SCREEN_EM) {
                            const float lost = (float)(v - (double)(float)v);
                            if (j0 == 0) dv = lost;
                            else val[off + j0 + l8] = lost;
                        }
                    }
                }
                __syncwarp();
                // the eight lanes of a point: its values, eight at a time
                float mx = -CUDART_INF_F;
                int best = 0x7fffffff;
                for (int j = l8; j < cnt; j += 8) {
                    const float l = pv[j];
                    if (MODE == SCREEN_ARGMAX) {
                        const int k = pk[j];
                        if (l > mx || (l == mx && k < best)) { mx = l; best = k; }
                    } else mx = fmaxf(mx, l);
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    const float om = __shfl_xor_sync(0xffffffffu, mx, o);
                    if (MODE == SCREEN_ARGMAX) {
                        const int ob = __shfl_xor_sync(0xffffffffu, best, o);
                        if (om > mx || (om == mx && ob < best)) { mx = om; best = ob; }
                    } else mx = fmaxf(mx, om);
                }
                if (MODE == SCREEN_ARGMAX) {
                    int near_n = 0;                                  // candidates within rounding of the best
                    const float near = 4e-6f * (fabsf(mx) + 300.f * __ldg(w2));      // (w2: the unit mixture's weight, see above)
                    for (int j = l8; j < cnt; j += 8) near_n += pv[j] >= mx - near ? 1 : 0;
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) near_n += __shfl_xor_sync(0xffffffffu, near_n, o);
                    for (unsigned ties = __ballot_sync(0xffffffffu, l8 == 0 && near_n > 1); ties; ties &= ties - 1) {
                        const int src = __ffs(ties) - 1;
                        const int at = __shfl_sync(0xffffffffu, (int)pt.y, src), n_c = __shfl_sync(0xffffffffu, cnt, src);
                        const float top_v = __shfl_sync(0xffffffffu, mx, src), band = __shfl_sync(0xffffffffu, near, src);
                        const int r = __shfl_sync(0xffffffffu, (int)pt.x, src);
                        const int k = screen_nearest(top.tie, X + (first + r) * D, D, mu, v_s + at, k_s + at, n_c, top_v, band, lane);
                        if (lane == src) best = k;
                    }
                    if (have && l8 == 0) {
                        if (idx) idx[prow] = best;
                        if (histogram) {
                            ids[off] = (unsigned short)best;
                            val[off] = -1.f;
                            pt_cnt[prow] = 1;
                            atomicAdd(&hist[best], 1);
                        }
                    }
                    continue;
                }
                float sum = 0.f;
                for (int j = l8; j < cnt; j += 8) sum += fast_ex2(pv[j] - mx);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                const float ls = log2f(sum), lz = mx + ls;
                if (MODE == SCREEN_TOP) {
                    float lv = CUDART_INF_F;                     // the pair that went out last
                    int lk = -1;
                    for (int r = 0; r < top.m; ++r) {
                        float bv = -CUDART_INF_F;
                        int bk = 0x7fffffff;
                        for (int j = l8; j < cnt; j += 8) {
                            const float v = pv[j];
                            const int k = pk[j];
                            if ((v < lv || (v == lv && k > lk)) && (v > bv || (v == bv && k < bk))) { bv = v; bk = k; }
                        }
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) {
                            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
                            const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                            if (ov > bv || (ov == bv && ok < bk)) { bv = ov; bk = ok; }
                        }
                        if (have && l8 == 0) {
                            idx[prow * top.m + r] = bk == 0x7fffffff ? 0 : bk;
                            if (top.resp) top.resp[prow * top.m + r] = fast_ex2(bv - lz);
                        }
                        lv = bv;
                        lk = bk;
                    }
                    continue;
                }
                if (have && l8 == 0) {
                    const double z = (double)mx + (double)ls;
                    if (MODE == SCREEN_LOGP) logp[prow] = (float)(z * 0.69314718055994530942);
                    ll_acc += z;
                }
                if (MODE == SCREEN_EM) {
                    // responsibilities; the pairs below 2^-40 of the total leave the list.  (The derivative of log Z by a pair's value is its responsibility.)
                    int kept = 0;
                    for (int j0 = 0; j0 < steps; j0 += 8) {
                        const int j = j0 + l8;
                        const float v = j < cnt ? pv[j] : -CUDART_INF_F, r = fast_ex2((v - mx) - ls);
                        const bool keep = r >= 9.094947e-13f;
                        if (j0 > 0) {
                            if (j < cnt) dv = val[off + j];
                            __syncwarp();
                        }
                        if (keep) ll_acc += (double)(r * dv);
                        const unsigned mine = (__ballot_sync(0xffffffffu, keep) >> (8 * grp)) & 255u;
                        if (keep) {
                            const unsigned short id = pk[j];
                            const int q = kept + __popc(mine & ((1u << l8) - 1u));
                            ids[off + q] = id;
                            val[off + q] = r;
                            if (histogram) atomicAdd(&hist[id], 1);
                        }
                        kept += __popc(mine);
                    }
                    if (have && l8 == 0) pt_cnt[prow] = kept;
                }
            }
            __syncwarp();
        }
        if (MODE == SCREEN_EM || MODE == SCREEN_LOGP) {
            ll_acc = warp_sum(ll_acc);
            if (lane == 0) ll_s[bt] = ll_acc;
        }
    }
    __syncthreads();
    if (histogram)
        for (int k = tid; k < K; k += 256) counts[(size_t)blockIdx.x * K + k] = hist[k];
    if ((MODE == SCREEN_EM || MODE == SCREEN_LOGP) && ll && warp == 0) {
        double s = lane < 8 ? red_s[lane] : 0.0;
        for (int b = lane; b < batches; b += 32) s += ll_s[b];
        s = warp_sum(s);
        if (lane == 0) ll[blockIdx.x] = s * 0.69314718055994530942 + ll[blockIdx.x];      // one owner per slot: launches add up
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Sort by component.  counts[b][k] -> where range b starts among component k's pairs; the last CTA to finish turns the totals
// into offsets and work items of SCR_SEG pairs.
__global__ void __launch_bounds__(1024) screen_scan_kernel(int* __restrict__ counts, int blocks, int K, int* __restrict__ totals,
                                                           int* __restrict__ off, int* __restrict__ segoff, int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    __shared__ int part[32][33];
    __shared__ int last_s;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int k = blockIdx.x * 32 + lane;
    const int per = (blocks + 31) / 32;
    const int b0 = min(blocks, w * per), b1 = min(blocks, b0 + per);
    int s = 0;
    if (k < K) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) s += counts[(size_t)b * K + k];
    }
    part[w][lane] = s;
    __syncthreads();
    int run = 0, total = 0;
    for (int j = 0; j < 32; ++j) {
        if (j < w) run += part[j][lane];
        total += part[j][lane];
    }
    if (k < K) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) {
            const int c = counts[(size_t)b * K + k];
            counts[(size_t)b * K + k] = run;
            run += c;
        }
        if (w == 0) totals[k] = total;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) last_s = atomicAdd(ctl + SC_TICKET_B, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    __shared__ int ws[2][32];
    int carry = 0, scarry = 0;
    for (int base = 0; base < K; base += 1024) {
        const int kk = base + tid;
        const int v = kk < K ? __ldcg(totals + kk) : 0, sv = (v + SCR_SEG - 1) / SCR_SEG;
        int inc = v, sinc = sv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, inc, o), b = __shfl_up_sync(0xffffffffu, sinc, o);
            if (lane >= o) { inc += a; sinc += b; }
        }
        if (lane == 31) { ws[0][w] = inc; ws[1][w] = sinc; }
        __syncthreads();
        int before = carry, sbefore = scarry, tot = 0, stot = 0;
        for (int j = 0; j < 32; ++j) {
            if (j < w) { before += ws[0][j]; sbefore += ws[1][j]; }
            tot += ws[0][j];
            stot += ws[1][j];
        }
        if (kk < K) {
            off[kk] = before + inc - v;
            segoff[kk] = sbefore + sinc - sv;
        }
        carry += tot;
        scarry += stot;
        __syncthreads();
    }
    if (tid == 0) {
        off[K] = carry;
        segoff[K] = scarry;
        ctl[SC_TICKET_B] = 0;
        const long long kept = (long long)ctl[SC_KEPT] + carry;
        ctl[SC_KEPT] = kept > 0x7fffffff ? 0x7fffffff : (int)kept;
    }
}

// A CTA per range, a warp per part of it (whole rounds of 32 points), with cursors of its own: lanes = points, their pairs one after the other,
// the pairs of one component ranked by lane.  The order is the same in every run.
__global__ void __launch_bounds__(1024) screen_fill_kernel(int64_t n, int K, int range, const unsigned* __restrict__ pt_off, const int* __restrict__ pt_cnt,
                                                           const unsigned short* __restrict__ ids, const float* __restrict__ val,
                                                           const int* __restrict__ starts, const int* __restrict__ off,
                                                           uint2* __restrict__ srt, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    extern __shared__ int sm[];                      // base [K], then the warps' cursors [W][K rounded up to even] as 16-bit values
    const int K2 = (K + 1) & ~1, W = blockDim.x >> 5;
    int* base = sm;
    unsigned* cur32 = reinterpret_cast<unsigned*>(sm + K2);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned short* cur = reinterpret_cast<unsigned short*>(cur32) + (size_t)warp * K2;
    for (int k = tid; k < K; k += blockDim.x) base[k] = __ldg(off + k) + starts[(size_t)blockIdx.x * K + k];
    for (int k = tid; k < W * K2 / 2; k += blockDim.x) cur32[k] = 0u;
    __syncthreads();
    const int part = ((range + W - 1) / W + 31) / 32 * 32;
    const int64_t p0 = (int64_t)blockIdx.x * range, end = p0 + range < n ? p0 + range : n;
    const int64_t w0 = p0 + warp * part, w1 = w0 + part < end ? w0 + part : end;
    for (int64_t row = w0 + lane; row < w1; row += 32) {
        const int c = pt_cnt[row];
        const unsigned o = pt_off[row];
        for (int j = 0; j < c; ++j) {
            const int k = ids[o + j];
            atomicAdd(cur32 + ((size_t)warp * K2 + k) / 2, 1u << (16 * (k & 1)));
        }
    }
    __syncthreads();
    for (int k = tid; k < K; k += blockDim.x) {
        unsigned c = 0;
        unsigned short* q = reinterpret_cast<unsigned short*>(cur32) + k;
#pragma unroll 8
        for (int w = 0; w < W; ++w) { const unsigned v = q[(size_t)w * K2]; q[(size_t)w * K2] = (unsigned short)c; c += v; }
    }
    __syncthreads();
    for (int64_t r0 = w0; r0 < w1; r0 += 32) {
        const int64_t row = r0 + lane;
        const int cnt = row < w1 ? pt_cnt[row] : 0;
        const unsigned o = row < w1 ? pt_off[row] : 0u;
        const int most = __reduce_max_sync(0xffffffffu, (unsigned)cnt);
        for (int j = 0; j < most; ++j) {
            const bool on = j < cnt;
            const int k = on ? ids[o + j] : -1;
            const float r = on ? val[o + j] : 0.f;
            const unsigned peers = __match_any_sync(0xffffffffu, k);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            int c = 0;
            if (on) c = cur[k];
            __syncwarp();
            if (on) {
                if (rank == 0) cur[k] = (unsigned short)(c + __popc(peers));
                srt[base[k] + c + rank] = make_uint2((unsigned)row, __float_as_uint(r));
            }
            __syncwarp();
        }
    }
}

// Statistics: sums of r, r (x - mu), r (x - mu)^2, and over the points whose only pair this is (r < 0) their number and sum_d w2 (x - mu)^2, which is their
// log-likelihood; fp32 within a work item (at most SCR_SEG pairs of one component), float64 beyond.  A warp takes as
// many consecutive items as make one wave of warps (screen_item_group); their pairs are neighbours in srt, whatever their components, so their rows come in one
// stream: ST_STAGES stages of ST_ROWS loads per lane, by asynchronous copies into shared memory, and the pairs themselves 32 ahead.  LPR lanes per row, four
// dimensions each; a stage that holds the end of an item is gone through once more for the next one.  A group g has one set of sums per component k in it, at
// place g + k (a later set has a larger g or a larger k).
// Bound by the gathered rows: 606K points at 128 x 1024, 1.36M rows, 140 us with four rows in flight per warp, 24 warps per SM, 60 instructions per row and a CTA's
// warps waiting for one another after 64 rows each (54 % of the issue slots, 3.6 TB/s from memory); 113 with eight rows in flight, no waiting and 20
// instructions (31 %, 4.3 TB/s).  A step of 1.02M x 128, K = 1024 with those 1036 us, with this 982, 12 warps per SM with 24 rows each on their way; with
// 16 warps and 16 rows 1030, 8 warps and 40 rows 994, four rows per stage 1065, and the pairs one stage ahead instead of 32 pairs 1075 to 1284.
// The log-likelihood of the points with several pairs is not sum_k r_k log z_k of these sums: 32 bits lose weights of 1e-8 beside others, each of which is as much of the
// log-likelihood as its log-density is of a point's (120K x 128, K = 1024: 1.7e-9 of it, against 5e-11).
constexpr int ST_ROWS = 8, ST_STAGES = 4;
__device__ __forceinline__ int screen_item_group(int items) { return items <= SCR_STAT_WARPS ? 1 : (items + SCR_STAT_WARPS - 1) / SCR_STAT_WARPS; }
// The component whose items hold this one: the last with segoff <= item.  The whole warp.
__device__ __forceinline__ int screen_component(const int* __restrict__ segoff, int K, int item, int lane) {
    int k = 0;
    for (int step = K > 1024 ? 1024 : K > 32 ? 32 : 1, span = K; ; step = step > 32 ? 32 : 1) {
        const int c = k + lane * step;
        const unsigned in = __ballot_sync(0xffffffffu, lane * step < span && __ldg(segoff + (lane * step < span ? c : k)) <= item);
        k += (31 - __clz(in | 1u)) * step;
        if (step == 1) return k;
        span = min(step, K - k);
    }
}
template <int LPR, bool VEC>
__global__ void __launch_bounds__(ST_THREADS, ST_CTAS) screen_stats_kernel(const float* __restrict__ X, int D, const float* __restrict__ mu,
                                                           const float* __restrict__ w2, const double* __restrict__ c2d,
                                                           const uint2* __restrict__ srt, const int* __restrict__ off, const int* __restrict__ segoff,
                                                           int K, double* __restrict__ part, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    constexpr int ROWS = 32 / LPR, U = LPR < ST_ROWS ? LPR : ST_ROWS, SR = U * ROWS;        // pairs of a stage (at most 32)
    constexpr int W = ST_THREADS / 32;
    extern __shared__ __align__(16) unsigned char ring_s[];                                 // [W][ST_STAGES][ST_ROWS][32] 16 bytes
    __shared__ double t_s[W][8][32];                 // a lane's sums of the items so far (x - mu: four dimensions, squares)
    __shared__ float r_s[W][ST_STAGES][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % LPR, sub = lane / LPR, d0 = 4 * l;
    const int items = __ldg(segoff + K), G = screen_item_group(items), g = blockIdx.x * W + warp;
    if (g * G >= items) return;
    const int first = g * G, end = min(items, first + G);
    double (*const t)[32] = t_s[warp];
    uint4* const ring = reinterpret_cast<uint4*>(ring_s) + (size_t)warp * ST_STAGES * ST_ROWS * 32 + lane;
    int k = screen_component(segoff, K, first, lane);
    const int p0 = __ldg(off + k) + (first - __ldg(segoff + k)) * SCR_SEG;
    int total;                                       // pairs of the group
    if (end == items) total = __ldg(off + K) - p0;
    else {
        const int ke = screen_component(segoff, K, end, lane);
        total = __ldg(off + ke) + (end - __ldg(segoff + ke)) * SCR_SEG - p0;
    }
    const int stages = (total + SR - 1) / SR;
    const uint2* const pairs = srt + p0;
    const float* const Xl = X + d0;
    uint2 e, e_next;                                 // 32 pairs of which the next stages are, and the 32 after them (no pair: row 0, without weight)
    auto fetch = [&](int i) {
        e_next = make_uint2(0u, 0u);
        if (i + lane < total) e_next = __ldg(pairs + i + lane);
    };
    auto issue = [&](int st) {
        const int slot = st % ST_STAGES, at = (st * SR) & 31;
        if (st < stages) {
            if (at == 0) {
                e = e_next;
                fetch(st * SR + 32);
            }
            const float r = __shfl_sync(0xffffffffu, __uint_as_float(e.y), (at + lane) & 31);
            if (lane < SR) r_s[warp][slot][lane] = r;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned row = __shfl_sync(0xffffffffu, e.x, at + u * ROWS + sub);
                const float* src = Xl + (size_t)row * D;
                const uint32_t dst = smem_u32(ring + (slot * ST_ROWS + u) * 32);
                if (VEC) {
                    if (d0 < D) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (d0 + j < D) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * j), "l"(src + j) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint64_t m[2];
    float w[4];
    int o1;
    auto component = [&]() {
        o1 = __ldg(off + k + 1) - p0;
        float f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            f[j] = d0 + j < D ? __ldg(mu + (size_t)k * D + d0 + j) : 0.f;
            w[j] = d0 + j < D ? __ldg(w2 + (size_t)k * D + d0 + j) : 0.f;
        }
        m[0] = pack2(__float_as_uint(f[0]), __float_as_uint(f[1]));
        m[1] = pack2(__float_as_uint(f[2]), __float_as_uint(f[3]));
    };
    fetch(0);
#pragma unroll 1
    for (int st = 0; st < ST_STAGES - 1; ++st) issue(st);
    component();
    int item = first, a = 0, b = min(SCR_SEG, o1);   // the item's pairs
    uint64_t s1[2] = {0ull, 0ull}, s2[2] = {0ull, 0ull}, q1[2] = {0ull, 0ull};               // (q1: squares of the points with one pair)
    float nsum = 0.f;
    int n1 = 0;
    double tn = 0.0, tq = 0.0;
    bool fresh = true;                               // the first item of a set of sums
#pragma unroll 1
    for (int st = 0; st < stages; ++st) {
        issue(st + ST_STAGES - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(ST_STAGES - 1) : "memory");
        __syncwarp();
        const int slot = st % ST_STAGES, pos = st * SR;
        const uint4* const xs = ring + slot * ST_ROWS * 32;
        const float* const rs = r_s[warp][slot];
        for (;;) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = pos + u * ROWS + sub;
                const bool on = i >= a && i < b;
                const float r = on ? rs[u * ROWS + sub] : 0.f;
                const uint4 x = xs[u * 32];
                const unsigned ra = __float_as_uint(fabsf(r)), r1 = r < 0.f ? 0x3F800000u : 0u;
                const uint64_t rr = pack2(ra, ra), one = pack2(r1, r1);
                uint64_t ta = sub2(pack2(x.x, x.y), m[0]), tb = sub2(pack2(x.z, x.w), m[1]);
                if (!on) ta = tb = 0ull;             // (a row of another component: the square may be beyond a float)
                s1[0] = fma2(rr, ta, s1[0]);
                s1[1] = fma2(rr, tb, s1[1]);
                ta = mul2(ta, ta);
                tb = mul2(tb, tb);
                s2[0] = fma2(rr, ta, s2[0]);
                s2[1] = fma2(rr, tb, s2[1]);
                q1[0] = fma2(one, ta, q1[0]);
                q1[1] = fma2(one, tb, q1[1]);
            }
            const float rl = lane < SR && pos + lane >= a && pos + lane < b ? rs[lane] : 0.f;
            nsum += fabsf(rl);
            n1 += rl < 0.f ? 1 : 0;
            if (b > pos + SR) break;
            // the item's last pair
            const float v[8] = {lo2(s1[0]), hi2(s1[0]), lo2(s1[1]), hi2(s1[1]), lo2(s2[0]), hi2(s2[0]), lo2(s2[1]), hi2(s2[1])};
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j][lane] = fresh ? (double)v[j] : t[j][lane] + (double)v[j];
            tn += (double)nsum;
            const float z[4] = {lo2(q1[0]), hi2(q1[0]), lo2(q1[1]), hi2(q1[1])};
            float q = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (d0 + j < D) q = fmaf(w[j], z[j], q);     // (beyond D garbage)
            tq += (double)q;
            fresh = false;
            s1[0] = s1[1] = s2[0] = s2[1] = q1[0] = q1[1] = 0ull;
            nsum = 0.f;
            a = b;
            ++item;
            if (b == o1 || item == end) {            // and the component's, or the group's
                double* const o = part + (size_t)(g + k) * (2 * D + 2);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    double q = t[j][lane];
#pragma unroll
                    for (int x = LPR; x < 32; x <<= 1) q += __shfl_xor_sync(0xffffffffu, q, x);
                    if (sub == 0 && d0 + (j & 3) < D) o[(j < 4 ? 0 : D) + d0 + (j & 3)] = q;
                }
                tn = warp_sum(tn);
                tq = warp_sum((n1 > 0 ? (double)n1 * __ldg(c2d + k) : 0.0) - tq);
                if (lane == 0) { o[2 * D] = tn; o[2 * D + 1] = tq; }
                if (item == end) break;
                do { ++k; } while (__ldg(segoff + k + 1) == item);               // (components without pairs)
                component();
                tn = tq = 0.0;
                n1 = 0;
                fresh = true;
            }
            b = min(a + SCR_SEG, o1);
            if (a >= pos + SR) break;
        }
        __syncwarp();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// A CTA per component: its sets of sums in order (two interleaved chains), float64, shifted from its mean to the origin.
__global__ void __launch_bounds__(512) screen_reduce_kernel(int D, int K, const double* __restrict__ part, const int* __restrict__ segoff,
                                                            const float* __restrict__ mu,
                                                            double* __restrict__ Nk, double* __restrict__ S1, double* __restrict__ S2,
                                                            double* __restrict__ llk, int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[SC_DONE] += 1;
    const int k = blockIdx.x, d = threadIdx.x & 127, q = (threadIdx.x >> 7) & 1, c = threadIdx.x >> 8;
    const int i0 = segoff[k], i1 = segoff[k + 1], G = screen_item_group(segoff[K]);
    if (i0 == i1) return;
    const int g0 = i0 / G + k, g1 = (i1 - 1) / G + k + 1;
    __shared__ double sh[2][2][128];
    __shared__ double tot[2];
    const size_t st = (size_t)(2 * D + 2);
    double a = 0.0;
    if (d < D)
        for (int g = g0 + c; g < g1; g += 8) {
            double v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = g + 2 * u < g1 ? part[(size_t)(g + 2 * u) * st + q * D + d] : 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u) a += v[u];
        }
    sh[c][q][d] = a;
    if (threadIdx.x < 64) {                              // warp: weight, log-likelihood of the points with one pair
        const int which = threadIdx.x >> 5, lane = threadIdx.x & 31;
        double t = 0.0;
        for (int g = g0 + lane; g < g1; g += 32) t += part[(size_t)g * st + 2 * D + which];
        t = warp_sum(t);
        if (lane == 0) tot[which] = t;
    }
    __syncthreads();
    if (threadIdx.x >= 128) return;
    const double n = tot[0];
    if (d < D) {
        const double s1 = sh[0][0][d] + sh[1][0][d], s2 = sh[0][1][d] + sh[1][1][d];
        const double m = (double)__ldg(mu + (size_t)k * D + d);
        S1[(size_t)k * D + d] += s1 + m * n;
        S2[(size_t)k * D + d] += s2 + 2.0 * m * s1 + m * m * n;
    }
    if (d == 0) {
        Nk[k] += n;
        llk[k] += tot[1] * 0.69314718055994530942;
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Groups of consecutive points (Fisher vectors): a CTA per group sorts the group's pairs by component (as screen_fill_kernel
// does for a range), the list in the group's own part of srt.
__global__ void __launch_bounds__(1024) screen_group_sort_kernel(int K, const int* __restrict__ g_start, const int* __restrict__ g_len,
                                                                const unsigned* __restrict__ pt_off, const int* __restrict__ pt_cnt,
                                                                const unsigned short* __restrict__ ids, const float* __restrict__ val,
                                                                int* __restrict__ g_off, uint2* __restrict__ srt, int* __restrict__ ctl) {
    if (screen_off(ctl)) return;
    extern __shared__ int sm[];                      // base [K], then the warps' cursors [W][K rounded up to even] as 16-bit values
    __shared__ int wsum[32];
    const int K2 = (K + 1) & ~1;
    int* base = sm;
    unsigned* cur32 = reinterpret_cast<unsigned*>(sm + K2);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5, g = blockIdx.x;
    unsigned short* cur = reinterpret_cast<unsigned short*>(cur32) + (size_t)warp * K2;
    const int start = g_start[g], len = g_len[g];
    int* off = g_off + (size_t)g * (K + 1);
    for (int k = tid; k < W * K2 / 2; k += blockDim.x) cur32[k] = 0u;
    __syncthreads();
    const int part = ((len + W - 1) / W + 31) / 32 * 32;
    const int p0 = start + min(len, warp * part), p1 = start + min(len, (warp + 1) * part);
    for (int row = p0 + lane; row < p1; row += 32) {
        const int c = pt_cnt[row];
        const unsigned o = pt_off[row];
        for (int j = 0; j < c; ++j) {
            const int k = ids[o + j];
            atomicAdd(cur32 + ((size_t)warp * K2 + k) / 2, 1u << (16 * (k & 1)));
        }
    }
    __syncthreads();
    // every component's start: thread t takes the components [t per, (t + 1) per)
    const int per = (K + (int)blockDim.x - 1) / (int)blockDim.x, k0 = min(K, tid * per), k1 = min(K, k0 + per);
    int own = 0;
    for (int k = k0; k < k1; ++k) {
        unsigned short* q = reinterpret_cast<unsigned short*>(cur32) + k;
        int c = 0;
        for (int w = 0; w < W; ++w) { const int v = q[(size_t)w * K2]; q[(size_t)w * K2] = (unsigned short)c; c += v; }
        base[k] = c;
        own += c;
    }
    int inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int run = inc - own, total = 0;
    for (int w = 0; w < W; ++w) {
        if (w < warp) run += wsum[w];
        total += wsum[w];
    }
    const int first = start * SCR_SLOTS;             // the group's part of srt
    for (int k = k0; k < k1; ++k) {
        const int c = base[k];
        base[k] = first + run;
        off[k] = first + run;
        run += c;
    }
    if (tid == 0) off[K] = first + total;
    if (total > len * SCR_SLOTS) {                   // (the same in every thread)
        if (tid == 0) ctl[SC_DENSE] = 1;
        return;
    }
    __syncthreads();
    for (int r0 = p0; r0 < p1; r0 += 32) {
        const int row = r0 + lane;
        const int c = row < p1 ? pt_cnt[row] : 0;
        const unsigned o = row < p1 ? pt_off[row] : 0u;
        const int most = __reduce_max_sync(0xffffffffu, (unsigned)c);
        for (int j = 0; j < most; ++j) {
            const bool on = j < c;
            const int k = on ? ids[o + j] : -1;
            const float r = on ? val[o + j] : 0.f;
            const unsigned peers = __match_any_sync(0xffffffffu, k);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            int q = 0;
            if (on) q = cur[k];
            __syncwarp();
            if (on) {
                if (rank == 0) cur[k] = (unsigned short)(q + __popc(peers));
                srt[base[k] + q + rank] = make_uint2((unsigned)row, __float_as_uint(r));
            }
            __syncwarp();
        }
    }
}

// Fisher vectors.  With sums about the component's mean,
//   G_mu = sum r (x - mu) / (T sigma sqrt(pi)),   G_sigma = (sum r (x - mu)^2 / var - sum r) / (T sqrt(2 pi)):
// nothing cancels.  fp32 sums of at most 32 pairs (however few a stage has) at a time, added in fp32, the weights in float64.  A warp has runs of GS_COMPS components of a group, whose pairs are neighbours: their rows
// come in one stream, as in screen_stats_kernel (GS_STAGES stages of GS_ROWS loads per lane), the parameters one component ahead.
// Bound by the gathered rows and the runs' first trips.  150 groups of 6827 points, us per call, with a warp per component and 16 rows in flight, waited for / now:
// 64 x 256 676 / 619, 128 x 512 1139 / 996, 100 x 33 881 / 682; 500 groups of 2000 x 64, K = 256 691 / 645.
constexpr int GS_COMPS = 8, GS_ROWS = 4, GS_STAGES = 8;      // (components of a run at most)
template <int LPR, bool VEC>
__global__ void __launch_bounds__(ST_THREADS, ST_CTAS) screen_group_stats_kernel(const float* __restrict__ X, int D, int K, int groups, int comps,
                                                                 const float* __restrict__ pi, const float* __restrict__ mu,
                                                                 const float* __restrict__ var, const float* __restrict__ w2,
                                                                 const double* __restrict__ c2d, const uint2* __restrict__ srt,
                                                                 const int* __restrict__ g_off, const int* __restrict__ g_len,
                                                                 float* __restrict__ fv, double* __restrict__ ll, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    constexpr int ROWS = 32 / LPR, U = LPR < GS_ROWS ? LPR : GS_ROWS, SR = U * ROWS;        // pairs of a stage (at most 32)
    constexpr int W = ST_THREADS / 32;
    static_assert(GS_COMPS < 32, "a lane per offset");
    extern __shared__ __align__(16) unsigned char ring_s[];                                 // [W][GS_STAGES][GS_ROWS][32] 16 bytes
    __shared__ float2 r_s[W][GS_STAGES][32];                                                // |r|; 1 where it is the point's only pair
    __shared__ double red[W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % LPR, sub = lane / LPR, d0 = 4 * l;
    uint4* const ring = reinterpret_cast<uint4*>(ring_s) + (size_t)warp * GS_STAGES * GS_ROWS * 32 + lane;
    const bool vec_o = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(fv) & 15) == 0);
    const bool vec_m = (D % 4 == 0) && (((reinterpret_cast<uintptr_t>(mu) | reinterpret_cast<uintptr_t>(var)) & 15) == 0);
    const size_t KD = (size_t)K * D;
    auto load4 = [&](const float* __restrict__ r, bool v) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v) {
            if (d0 < D) a = __ldg(reinterpret_cast<const float4*>(r + d0));
        } else {
            if (d0 < D) a.x = __ldg(r + d0);
            if (d0 + 1 < D) a.y = __ldg(r + d0 + 1);
            if (d0 + 2 < D) a.z = __ldg(r + d0 + 2);
            if (d0 + 3 < D) a.w = __ldg(r + d0 + 3);
        }
        return a;
    };
    struct Comp { float4 m, w, v; float p; };
    auto component = [&](int k) {
        Comp c;
        c.m = load4(mu + (size_t)k * D, vec_m);
        c.v = load4(var + (size_t)k * D, vec_m);
        c.w = load4(w2 + (size_t)k * D, (D & 3) == 0);       // (scratch, aligned)
        c.p = __ldg(pi + k);
        return c;
    };
    double ll_acc = 0.0;
    const float* const Xl = X + d0;
    const int per = (K + comps - 1) / comps, runs = groups * per;        // (at most 2^23)
#pragma unroll 1
    for (int run = blockIdx.x * W + warp; run < runs; run += gridDim.x * W) {
        const int g = run / per, k0 = (run - g * per) * comps, k1 = min(K, k0 + comps);
        const int o = __ldg(g_off + (size_t)g * (K + 1) + k0 + min(lane, k1 - k0));
        Comp c = component(k0);
        const int p0 = __shfl_sync(0xffffffffu, o, 0), total = __shfl_sync(0xffffffffu, o, k1 - k0) - p0, stages = (total + SR - 1) / SR;
        const uint2* const pairs = srt + p0;
        const float inv_t = 1.0f / (float)__ldg(g_len + g);
        uint2 e = make_uint2(0u, 0u), e_next;                // 32 pairs of which the next stages are, and the 32 after them (no pair: row 0, without weight)
        auto fetch = [&](int i) {
            e_next = make_uint2(0u, 0u);
            if (i + lane < total) e_next = __ldg(pairs + i + lane);
        };
        auto issue = [&](int st) {
            const int slot = st % GS_STAGES, at = (st * SR) & 31;
            if (st < stages) {
                if (at == 0) {
                    e = e_next;
                    fetch(st * SR + 32);
                }
                const float r = __shfl_sync(0xffffffffu, __uint_as_float(e.y), (at + lane) & 31);
                if (lane < SR) r_s[warp][slot][lane] = make_float2(fabsf(r), r < 0.f ? 1.f : 0.f);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned row = __shfl_sync(0xffffffffu, e.x, at + u * ROWS + sub);
                    const float* src = Xl + (size_t)row * D;
                    const uint32_t dst = smem_u32(ring + (slot * GS_ROWS + u) * 32);
                    if (VEC) {
                        if (d0 < D) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (d0 + j < D) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * j), "l"(src + j) : "memory");
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0);
#pragma unroll 1
        for (int st = 0; st < GS_STAGES - 1; ++st) issue(st);
        int cur = 0, ready = -1;                             // pairs done; the stage that has arrived
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            const int b = __shfl_sync(0xffffffffu, o, k - k0 + 1) - p0;
            const Comp now = c;
            if (k + 1 < k1) c = component(k + 1);
            uint64_t m[2] = {pack2(__float_as_uint(now.m.x), __float_as_uint(now.m.y)), pack2(__float_as_uint(now.m.z), __float_as_uint(now.m.w))};
            float s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f}, fn = 0.f;
            uint64_t f1[2] = {0ull, 0ull}, f2[2] = {0ull, 0ull}, q1[2] = {0ull, 0ull};           // (of the 32 pairs at hand, as fn; q1: of the points with one pair)
            const float va[4] = {now.v.x, now.v.y, now.v.z, now.v.w}, wa[4] = {now.w.x, now.w.y, now.w.z, now.w.w};
            float n1 = 0.f;
            double nsum = 0.0;
            const bool any = cur < b;
#pragma unroll 1
            while (cur < b) {
                const int st = cur / SR, pos = st * SR, to = min(b, pos + SR), slot = st % GS_STAGES;
                if (st != ready) {
                    __syncwarp();                            // (the stage before has been read)
                    issue(st + GS_STAGES - 1);
                    asm volatile("cp.async.wait_group %0;" ::"n"(GS_STAGES - 1) : "memory");
                    __syncwarp();
                    ready = st;
                }
                const uint4* const xs = ring + slot * GS_ROWS * 32;
                const float2* const rs = r_s[warp][slot];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = pos + u * ROWS + sub;
                    const bool on = i >= cur && i < to;
                    const float2 r = rs[u * ROWS + sub];
                    const uint4 x = xs[u * 32];
                    const uint64_t rr = pack2(__float_as_uint(r.x), __float_as_uint(r.x)), one = pack2(__float_as_uint(r.y), __float_as_uint(r.y));
                    uint64_t ta = sub2(pack2(x.x, x.y), m[0]), tb = sub2(pack2(x.z, x.w), m[1]);
                    if (!on) ta = tb = 0ull;                 // (a row of another component: the square may be beyond a float)
                    f1[0] = fma2(rr, ta, f1[0]);
                    f1[1] = fma2(rr, tb, f1[1]);
                    ta = mul2(ta, ta);
                    tb = mul2(tb, tb);
                    f2[0] = fma2(rr, ta, f2[0]);
                    f2[1] = fma2(rr, tb, f2[1]);
                    q1[0] = fma2(one, ta, q1[0]);
                    q1[1] = fma2(one, tb, q1[1]);
                }
                if (lane < SR && pos + lane >= cur && pos + lane < to) {
                    fn += rs[lane].x;
                    n1 += rs[lane].y;
                }
                cur = to;
                if (to == b || (to & 31) == 0) {
                    s1[0] += lo2(f1[0]); s1[1] += hi2(f1[0]); s1[2] += lo2(f1[1]); s1[3] += hi2(f1[1]);
                    s2[0] += lo2(f2[0]); s2[1] += hi2(f2[0]); s2[2] += lo2(f2[1]); s2[3] += hi2(f2[1]);
                    nsum += (double)fn;
                    const float z[4] = {lo2(q1[0]), hi2(q1[0]), lo2(q1[1]), hi2(q1[1])};
                    float q = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (d0 + j < D) q = fmaf(wa[j], z[j], q);        // (beyond D garbage)
                    ll_acc -= (double)q;
                    f1[0] = f1[1] = f2[0] = f2[1] = q1[0] = q1[1] = 0ull;
                    fn = 0.f;
                }
            }
            float gm[4] = {0.f, 0.f, 0.f, 0.f}, gs[4] = {0.f, 0.f, 0.f, 0.f};
            if (any) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int x = LPR; x < 32; x <<= 1) {
                        s1[j] += __shfl_xor_sync(0xffffffffu, s1[j], x);
                        s2[j] += __shfl_xor_sync(0xffffffffu, s2[j], x);
                    }
                if (n1 > 0.f) ll_acc += (double)n1 * __ldg(c2d + k);
                float nk = (float)nsum;
#pragma unroll
                for (int x = 16; x > 0; x >>= 1) nk += __shfl_xor_sync(0xffffffffu, nk, x);
                const float wk = now.p;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (wk > 0.f && d0 + j < D) {
                        gm[j] = s1[j] * (inv_t * rsqrtf(va[j]) * rsqrtf(wk));
                        gs[j] = (s2[j] - nk * va[j]) * (inv_t * rsqrtf(2.0f * wk) / va[j]);
                    }
            }
            if (sub == 0 && d0 < D) {
                float* out = fv + (size_t)g * 2 * KD + (size_t)k * D + d0;
                if (vec_o) {
                    *reinterpret_cast<float4*>(out) = make_float4(gm[0], gm[1], gm[2], gm[3]);
                    *reinterpret_cast<float4*>(out + KD) = make_float4(gs[0], gs[1], gs[2], gs[3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (d0 + j < D) { out[j] = gm[j]; out[KD + j] = gs[j]; }
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
    ll_acc = warp_sum(ll_acc);
    if (lane == 0) red[warp] = ll_acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < W; ++w) t += red[w];
        ll[blockIdx.x] += t * 0.69314718055994530942;
    }
}

// k-means: the centroids' new positions from their sums (a centroid without points stays), the points per centroid, the inertia
// per centroid (sum of -log2 z of its points).
__global__ void __launch_bounds__(128) screen_centroids_kernel(int D, int K, const float* __restrict__ cent_in, const double* __restrict__ Nk,
                                                               const double* __restrict__ S1, const double* __restrict__ llk,
                                                               float* __restrict__ cent_out, int64_t* __restrict__ counts,
                                                               double* __restrict__ inertia_k, const float* __restrict__ sd, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    const int k = blockIdx.x, d = threadIdx.x;
    const float F = d < 32 ? screen_unit_weight(D, sd, d) : 1.f;
    const double n = Nk[k];
    if (d < D) cent_out[(size_t)k * D + d] = n > 0.0 ? (float)(S1[(size_t)k * D + d] / n) : cent_in[(size_t)k * D + d];
    if (d == 0) {
        if (counts) counts[k] = (int64_t)(n + 0.5);
        inertia_k[k] = -llk[k] / (0.69314718055994530942 * (double)F);
    }
}

#define LCHECK()                                       \
    do {                                               \
        const cudaError_t e_ = cudaGetLastError();     \
        if (e_ != cudaSuccess) return e_;              \
    } while (0)

}  // namespace

// Points per CTA of the evaluation and of the sort by component: as many as make one wave of the evaluation (three CTAs per SM; two waves of half the
// points: a step of 1M x 128, K = 1024 1159 us against 1084, two thirds of a wave 1123), at least 64, or 128 where the statistics sort them.
static int screen_range(int64_t n, bool count) {
    const int r = (int)((n + SCR_RANGES - 1) / SCR_RANGES + 31) / 32 * 32, least = count ? 128 : 64;
    return r < least ? least : r;
}
// Whether the evaluation sorts a CTA's points: with about 450 of them and more it pays (us, sorted / as they come: a step of 128 x 1024 on 100K, 200K,
// 300K points 228 / 220, 341 / 347, 399 / 418; top-2 of 64 x 512 174 / 164, 222 / 217, 267 / 269; scores of 96 x 512 143 / 141, 190 / 199, 226 / 238).
static bool screen_sorts(int64_t n) { return n > 200000; }

bool screen_supports(int D, int K) { return D >= 1 && D <= 128 && K >= 1 && K <= SCR_MAX_K; }

cudaError_t launch_screen_prepare(cudaStream_t s, int D, int K, const float* pi, const float* mu, const float* var, bool unit,
                                  const ScreenProbe& probe, const ScreenBuffers& b, float* w2, float* c2, double* c2d, int* status) {
    const int Kpad = screen_kpad(K);
    const int db = (K + 7) / 8 < SCR_DIM_BLOCKS ? (K + 7) / 8 : SCR_DIM_BLOCKS;
    screen_dim_kernel<<<db, 512, 0, s>>>(D, K, pi, mu, var, unit ? 1 : 0, b.dimpart, b.sd, b.gd, b.ctl);
    LCHECK();
    screen_comp_kernel<<<(K + 7) / 8, 256, 0, s>>>(D, K, pi, mu, var, unit ? 1 : 0, b.sd, b.gd, w2, c2, c2d, b.prm, b.key, b.blk, b.probe, b.ll, b.ctl, status);
    LCHECK();
    static_assert((size_t)PR_GROUPS * PR_ROWS * SCR_MAX_K <= (size_t)SCR_PAIRS, "the probe's bounds lie where the sorted pairs will");
    const ProbeArgs pr{probe, K, mu, w2, c2d, b.prm, b.key, b.probe, Kpad / 8, reinterpret_cast<float2*>(b.srt), b.ctl};
    screen_plane_kernel<<<Kpad / 8 + (probe.n > 0 ? PR_GROUPS * PR_CTAS : 0), 256, 0, s>>>(pr, D, K, Kpad, unit ? 1 : 0, mu, w2, b.sd, b.gd, b.prm, b.key, b.p, b.blk, b.comp_of);
    return cudaGetLastError();
}

cudaError_t launch_screen_sweep(cudaStream_t s, const float* X, int64_t n, int D, int K, bool unit, float margin, int top, float max_marks, bool stats,
                                const float* mu, const float* w2, const double* c2d, const ScreenBuffers& b, int* status, int sms,
                                int64_t* launches) {
    if (n < 1 || n > SCR_PIECE) return cudaErrorInvalidValue;
    const int KC = (D + 7) / 8, KS = unit ? (KC + 1) / 2 : KC;
    const int Kpad = screen_kpad(K), KA = screen_atoms(D, unit);
    SweepParams p;
    p.n = n; p.KA = KA; p.KS = KS; p.KC = KC; p.unit = unit; p.NG = Kpad / 128; p.margin = margin;
    p.chunks = screen_chunks(D); p.X = X; p.D = D; p.sd = b.sd; p.gd = b.gd; p.y = b.y; p.n2 = b.n2; p.img = b.p; p.gbytes = (int)screen_group_bytes(D, unit);
    p.blk = b.blk; p.pt_off = b.pt_off; p.pt_cnt = b.pt_cnt; p.words = b.words; p.spill = b.spill;
    p.ovf = b.ovf; p.ctl = b.ctl; p.status = status; p.test_silent = b.test_silent;
    if (top < 1 || top > 4) return cudaErrorInvalidValue;
    const bool convert = screen_converts(D, K);
    if (!convert) {
        if (D > 64) return cudaErrorInvalidValue;            // (the sweep that takes rows of u has room for 8 chunks)
        int L = 1;
        while (L < KC) L <<= 1;
        const int rpb = 256 / L;
        int64_t blocks = (n + 2 * rpb - 1) / (2 * rpb);
        if (blocks > (int64_t)sms * 8) blocks = (int64_t)sms * 8;
#define FG_TR(L_) screen_transform_kernel<L_><<<(unsigned)blocks, 256, 0, s>>>(X, n, D, screen_chunks(D), b.sd, b.gd, b.y, b.n2, b.ctl)
        switch (L) {
            case 1: FG_TR(1); break;
            case 2: FG_TR(2); break;
            case 4: FG_TR(4); break;
            default: FG_TR(8); break;
        }
#undef FG_TR
        LCHECK();
        ++*launches;
    }
    auto sweep = convert ? (top == 1 ? screen_sweep_kernel<1, true> : top == 2 ? screen_sweep_kernel<2, true> : screen_sweep_kernel<4, true>)
                         : (top == 1 ? screen_sweep_kernel<1, false> : top == 2 ? screen_sweep_kernel<2, false> : screen_sweep_kernel<4, false>);
    const int sweep_smem = convert ? Sweep<true>::SMEM : Sweep<false>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, sweep_smem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + SCR_TILE - 1) / SCR_TILE;
    if (sms > SCR_MAX_SMS) sms = SCR_MAX_SMS;
    sweep<<<(unsigned)(tiles < sms ? tiles : sms), convert ? Sweep<true>::THREADS : Sweep<false>::THREADS, sweep_smem, s>>>(p);
    LCHECK();
    const size_t smem = (size_t)OV_ROWS * K * 4;
    // (here and below the same limit from every call: it belongs to the kernel, which contexts on other threads launch for other K)
    e = cudaFuncSetAttribute(screen_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OV_ROWS * SCR_MAX_K * 4);
    if (e != cudaSuccess) return e;
    const double most = fmin((double)max_marks * (double)n, (double)SCR_PIECE * (stats ? SCR_MARKS : SCR_SLOTS));
    screen_rows_kernel<<<(unsigned)(2 * sms), 256, smem, s>>>(X, n, D, K, margin, top, (long long)most, mu, w2, c2d, b.ovf,
                                                              b.pt_off, b.pt_cnt, b.ids, b.ctl);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_screen_eval(cudaStream_t s, int mode, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                               const double* c2d, const ScreenBuffers& b, float* logp, int32_t* idx, bool count, int m, float* resp, const ScreenTie* tie) {
    // (ranges as launch_screen_stats has them)
    const int range = screen_range(n, count), sorted = screen_sorts(n) ? 1 : 0;
    const unsigned blocks = (unsigned)((n + range - 1) / range);
    const size_t smem_order = (size_t)range * 4, smem = (size_t)K * 4 + smem_order;
    int* counts = count ? b.counts : nullptr;
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0) && ((reinterpret_cast<uintptr_t>(mu) & 15) == 0) && ((reinterpret_cast<uintptr_t>(w2) & 15) == 0);
    const TopOut out{m, resp, tie ? *tie : ScreenTie{}};
#define FG_EVAL(M_, N_, V_)                                                                                                                       \
    do {                                                                                                                                         \
        const cudaError_t e_ = cudaFuncSetAttribute(screen_eval_kernel<M_, N_, V_>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCR_MAX_K * 4 + EV_RANGE * 4); \
        if (e_ != cudaSuccess) return e_;                                                                                                        \
        screen_eval_kernel<M_, N_, V_><<<blocks, 256, (M_ == SCREEN_EM || M_ == SCREEN_ARGMAX) ? smem : smem_order, s>>>(X, n, D, K, mu, w2, c2d, \
        b.comp_of, range, sorted, b.words, b.pt_off, b.pt_cnt, b.ids, b.val, counts, b.ll, logp, idx, b.ctl, out);                               \
    } while (0)
#define FG_EVALS(M_)                                                                                            \
    switch ((D + 31) / 32) {                                                                                    \
        case 1: if (vec) FG_EVAL(M_, 1, true); else FG_EVAL(M_, 1, false); break;                               \
        case 2: if (vec) FG_EVAL(M_, 2, true); else FG_EVAL(M_, 2, false); break;                               \
        case 3: if (vec) FG_EVAL(M_, 3, true); else FG_EVAL(M_, 3, false); break;                               \
        default: if (vec) FG_EVAL(M_, 4, true); else FG_EVAL(M_, 4, false); break;                              \
    }
    switch (mode) {
        case SCREEN_EM: FG_EVALS(SCREEN_EM) break;
        case SCREEN_LOGP: FG_EVALS(SCREEN_LOGP) break;
        case SCREEN_TOP: FG_EVALS(SCREEN_TOP) break;
        default: FG_EVALS(SCREEN_ARGMAX) break;
    }
#undef FG_EVALS
#undef FG_EVAL
    return cudaGetLastError();
}

// One thread: which kernels have the word.
__global__ void screen_gate_kernel(int* __restrict__ ctl, int* __restrict__ gate, int* __restrict__ fallback, long long p, int first) {
    if (first) ctl[SC_ILL] = gate == nullptr || *gate != 0 ? 1 : 0;
    const bool todo = ctl[SC_DENSE] != 0 && p >= ctl[SC_DONE], ill = ctl[SC_ILL] != 0;
    *fallback = todo && ill ? 1 : 0;
    if (gate) *gate = todo && !ill ? 0 : 1;
}
cudaError_t launch_screen_gate(cudaStream_t s, const ScreenBuffers& b, int* gate, int* fallback, int64_t p, bool first) {
    screen_gate_kernel<<<1, 1, 0, s>>>(b.ctl, gate, fallback, (long long)p, first ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_screen_stats(cudaStream_t s, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                                const double* c2d, const ScreenBuffers& b, double* Nk, double* S1, double* S2, int64_t* launches) {
    const int range = screen_range(n, true), blocks = (int)((n + range - 1) / range);
    screen_scan_kernel<<<(K + 31) / 32, 1024, 0, s>>>(b.counts, blocks, K, b.totals, b.off, b.segoff, b.ctl);
    LCHECK();
    const int K2 = (K + 1) & ~1;
    constexpr int FILL_CURSORS = 32768;                      // warps x components, 2 bytes each
    // (at most 16 warps, so that the CTAs are one wave, four per SM at K = 1024: 1.2M x 100 50 us with 16, 80 with 32 - one and a half waves)
    int warps = range / 32;
    while (warps > 8 && (warps > 16 || warps * K2 > FILL_CURSORS)) --warps;
    const size_t smem = (size_t)K2 * 4 + (size_t)K2 * 2 * warps;
    cudaError_t e = cudaFuncSetAttribute(screen_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SCR_MAX_K * 4 + 2 * FILL_CURSORS);
    if (e != cudaSuccess) return e;
    screen_fill_kernel<<<blocks, warps * 32, smem, s>>>(n, K, range, b.pt_off, b.pt_cnt, b.ids, b.val, b.counts, b.off, b.srt, b.ctl);
    LCHECK();
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0) && ((reinterpret_cast<uintptr_t>(mu) & 15) == 0);
#define FG_STATS(L_) (vec ? screen_stats_kernel<L_, true> : screen_stats_kernel<L_, false>)
    const auto stats = D <= 8 ? FG_STATS(2) : D <= 16 ? FG_STATS(4) : D <= 32 ? FG_STATS(8) : D <= 64 ? FG_STATS(16) : FG_STATS(32);
#undef FG_STATS
    constexpr int stats_smem = ST_THREADS / 32 * ST_STAGES * ST_ROWS * 512;
    e = cudaFuncSetAttribute(stats, cudaFuncAttributeMaxDynamicSharedMemorySize, stats_smem);
    if (e != cudaSuccess) return e;
    stats<<<SCR_STAT_WARPS / (ST_THREADS / 32), ST_THREADS, stats_smem, s>>>(X, D, mu, w2, c2d, b.srt, b.off, b.segoff, K, b.part, b.ctl);
    LCHECK();
    screen_reduce_kernel<<<K, 512, 0, s>>>(D, K, b.part, b.segoff, mu, Nk, S1, S2, b.ll + SCR_LL, b.ctl);
    *launches += 4;
    return cudaGetLastError();
}

cudaError_t launch_screen_groups(cudaStream_t s, const float* X, int64_t n, int groups, int D, int K, const int* g_start, const int* g_len, int* g_off,
                                 const float* pi, const float* mu, const float* var, const float* w2, const double* c2d,
                                 const ScreenBuffers& b, float* fv, int64_t* launches) {
    const int K2 = (K + 1) & ~1;
    constexpr int GROUP_CURSORS = 131072;                    // cursors of 2 bytes per warp and component: at most 128 KB
    int warps = 32;
    while (warps > 8 && (size_t)K2 * warps * 2 > GROUP_CURSORS) warps >>= 1;
    const size_t smem = (size_t)K2 * 4 + (size_t)K2 * warps * 2;
    cudaError_t e = cudaFuncSetAttribute(screen_group_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SCR_MAX_K * 4 + GROUP_CURSORS);
    if (e != cudaSuccess) return e;
    screen_group_sort_kernel<<<groups, warps * 32, smem, s>>>(K, g_start, g_len, b.pt_off, b.pt_cnt, b.ids, b.val, g_off, b.srt, b.ctl);
    LCHECK();
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
#define FG_GROUPS(L_) (vec ? screen_group_stats_kernel<L_, true> : screen_group_stats_kernel<L_, false>)
    const auto stats = D <= 8 ? FG_GROUPS(2) : D <= 16 ? FG_GROUPS(4) : D <= 32 ? FG_GROUPS(8) : D <= 64 ? FG_GROUPS(16) : FG_GROUPS(32);
#undef FG_GROUPS
    constexpr int stats_smem = ST_THREADS / 32 * GS_STAGES * GS_ROWS * 512;
    e = cudaFuncSetAttribute(stats, cudaFuncAttributeMaxDynamicSharedMemorySize, stats_smem);
    if (e != cudaSuccess) return e;
    // A run has about 400 pairs (2.2 kept ones per point on separate clusters), but there are runs enough for two rounds of warps: 150 groups of 6827, 64 x 256,
    // runs of 8, 16, 31 components 627, 660, 661 us, 100 x 33 795, 1100, 1468 and with one 659.
    const double pairs = 2.2 * (double)n / ((double)groups * K);
    int comps = pairs * GS_COMPS <= 400.0 ? GS_COMPS : pairs >= 400.0 ? 1 : (int)(400.0 / pairs);
    while (comps > 1 && (int64_t)groups * ((K + comps - 1) / comps) < 2 * SCR_STAT_WARPS) comps = (comps + 1) / 2;
    stats<<<SCR_STAT_WARPS / (ST_THREADS / 32), ST_THREADS, stats_smem, s>>>(X, D, K, groups, comps, pi, mu, var, w2, c2d, b.srt, g_off, g_len, fv, b.ll, b.ctl);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_screen_centroids(cudaStream_t s, int D, int K, const float* cent_in, const double* Nk, const double* S1,
                                    const ScreenBuffers& b, float* cent_out, int64_t* counts, double* inertia_k) {
    screen_centroids_kernel<<<K, 128, 0, s>>>(D, K, cent_in, Nk, S1, b.ll + SCR_LL, cent_out, counts, inertia_k, b.sd, b.ctl);
    return cudaGetLastError();
}

}  // namespace fg
