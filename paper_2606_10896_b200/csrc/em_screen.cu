// The screening path for D <= 128 (sm_100a, tcgen05 + TMEM): few (point, component) pairs of a mixture matter.
//
// Where posteriors are sparse - a handful of components within 2^-40 of a point's best - only those pairs need their exact
// densities and statistics.  ONE sweep of the tensor cores over a single fp16 product per contraction (a sixth of the work of
// the kernels that form every responsibility from split operands) tells which they are, with rigorous error bounds:
//
//   screen_sweep_kernel   TMEM lanes = points.  A CTA holds the fp16 plane of 256 points in shared memory and streams the
//                         components' coefficients past it, 128 at a time; a softmax thread owns one point, keeps the largest
//                         lower bound seen so far and the components whose upper bound reaches it (less the margin), drops
//                         those that the final bound rules out, and writes the rest as a list.
//   screen_eval_kernel    the listed pairs in fp32 direct differences: log-sum-exp, responsibilities, or the arg-max.
//   screen_scan/fill/stats/reduce   the kept pairs sorted by component (stable, no atomics on the output), streamed as rows of
//                         X against the component's mean in registers, fp32 within 64 pairs, float64 beyond.
//
// Every value that reaches a result comes from exact fp32 evaluations; a term below 2^-40 of a point's total is dropped.  Data
// whose posteriors are broad is noticed by the first sweep (SC_DENSE): the kernels that follow return at once and the caller
// runs the dense kernels instead.
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
// c = log2 pi + ... - sum_d b nu^2.  Rows are divided by a power of two t (largest coefficient in [512, 1024)) and rounded
// to fp16.
//
// Error of the approximate log2 z of ANY point: every product is formed from two operands rounded to 2^-11 (or to 2^-25, the
// spacing of subnormals) and added into an fp32 accumulator that loses less than 2^-18 of the terms' sizes, and the sizes add
// up to at most  sum_d b (2 |nu u| + u^2) <= sum_d b nu^2 + 2 max_d b |u|^2.  So it is below alpha + beta |u|^2 with
//   alpha = eps sum_d b nu^2 + 2^-24 sum_d (2 b |nu| + b) + t 2^-25 D / 2 + 2^-22 |c| + 0.02
//   beta  = 2 eps max_d b + 1.5 t 2^-25,        eps = 2^-10 (1 + 2^-6).
//
// A component that is much narrower than the data in some dimensions (a few points, one point) has a huge max_d b, and with it
// an allowance that rules nothing out.  Where the allowance of a typical point exceeds SCR_SHARP bits, b is CAPPED at a value
// that leaves about 16: c - sum_d min(b, cap) (u - nu)^2 is an upper bound of log2 z, which is what the screening needs, with a
// small allowance; only its lower bound is lost, so such components do not raise the threshold.
constexpr float SCR_SHARP = 40.f;
constexpr float SCR_CAPPED = 1e30f;          // their sorting key
__device__ __forceinline__ double screen_cap(int D) { return 16.0 / (2.0 * 9.765625e-04 * (double)D); }

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
        ctl[SC_TICKET_A] = 0;
        ctl[SC_DENSE] = 0;
        ctl[SC_ACTIVE] = 0;
        ctl[SC_KEPT] = 0;
    }
}

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

// A warp per component: the FP32 kernels' derived parameters, the row's scale and constant, and the allowances above.
__global__ void __launch_bounds__(256) screen_comp_kernel(int D, int K, const float* __restrict__ pi, const float* __restrict__ mu,
                                                          const float* __restrict__ var, int unit, const float* __restrict__ sd,
                                                          const float* __restrict__ gd, float* __restrict__ w2, float* __restrict__ c2,
                                                          double* __restrict__ c2d, float4* __restrict__ prm, float* __restrict__ key,
                                                          int4* __restrict__ blk, int* __restrict__ ctl, int* __restrict__ status) {
    const int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x < SCR_MAX_K / 32) blk[threadIdx.x] = make_int4(0, 0, 0, 0);      // (largest allowances, see below)
    if (k >= K) return;
    double slog = 0.0, bv[4], nv[4];
    int bad = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int d = lane + 32 * i;
        bv[i] = nv[i] = 0.0;
        if (d >= D) continue;
        const float v = unit ? 1.f : __ldg(var + (size_t)k * D + d), m = __ldg(mu + (size_t)k * D + d);
        if (!(v > 0.f) || !isfinite(v)) bad |= ST_BAD_VAR;
        if (!isfinite(m)) bad |= ST_NONFINITE;
        const double w = unit ? 1.0 : 0.72134752044448170368 / (double)v;
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
    double bnn, t, c, al, be;
    bool capped = false;
    for (;;) {                                       // (at most twice; the same way in every lane)
        double absab = 0.0, bmax = 0.0, cmax = 0.0;
        bnn = 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double b = capped ? fmin(bv[i], screen_cap(D)) : bv[i];
            bnn += b * nv[i] * nv[i];
            absab += 2.0 * b * fabs(nv[i]) + b;
            bmax = fmax(bmax, b);
            cmax = fmax(cmax, fmax(b, 2.0 * b * fabs(nv[i])));
        }
        bnn = warp_sum(bnn); absab = warp_sum(absab); bmax = warp_max(bmax); cmax = warp_max(cmax);
        t = 1.0;
        if (cmax > 0.0 && isfinite(cmax)) t = exp2(floor(log2(cmax)) - 9.0);
        c = cd - bnn;
        al = eps * bnn + 5.9604644775390625e-08 * absab + t * 2.98023223876953125e-08 * 0.5 * D + 2.384185791015625e-07 * fabs(c) + 0.02;
        be = 2.0 * eps * bmax + t * 2.98023223876953125e-08 * 1.5;
        if (capped || !(al + be * D > (double)SCR_SHARP)) break;
        capped = true;
    }
    if (lane == 0) {
        if (c2) c2[k] = (float)cd;
        c2d[k] = cd;
        const bool on = p > 0.f && isfinite(c) && isfinite(al) && isfinite(be);
        prm[k] = make_float4((float)t, on ? (float)c : -CUDART_INF_F, on ? (float)(al * 1.000001) : 0.f, on ? (float)(be * 1.000001) : 0.f);
        key[k] = !on ? CUDART_INF_F : capped ? SCR_CAPPED : (float)(al + be * D);
        if (on) atomicAdd(ctl + SC_ACTIVE, 1);
        if (bad) atomicOr(status, bad);
    }
}

// Positions of the components in the sweep: ascending by the allowance of a typical point, so that 32 neighbours, which are
// screened with the largest allowance among them, have similar ones (the capped components come last).  A warp per component:
// its rank among the keys is its position, and it writes its own row (a sort of the keys in every CTA took 20 us).
__global__ void __launch_bounds__(256) screen_plane_kernel(int D, int K, int Kpad, const float* __restrict__ mu,
                                                           const float* __restrict__ w2, const float* __restrict__ sd,
                                                           const float* __restrict__ gd, const float4* __restrict__ prm,
                                                           const float* __restrict__ key, __half* __restrict__ p, float4* __restrict__ tab,
                                                           int4* __restrict__ blk, int* __restrict__ comp_of) {
    const int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (k >= Kpad) return;
    int pos = k;
    bool on = false, capped = false;
    float4 q = make_float4(1.f, -CUDART_INF_F, 0.f, 0.f);
    if (k < K) {
        const float mine = __ldg(key + k);
        int before = 0;
#pragma unroll 8
        for (int j = lane; j < K; j += 32) {
            const float o = __ldg(key + j);
            before += (o < mine || (o == mine && j < k)) ? 1 : 0;
        }
        pos = __reduce_add_sync(0xffffffffu, before);
        on = mine < CUDART_INF_F;
        capped = on && mine >= SCR_CAPPED;
        if (on) q = __ldg(prm + k);
    }
    const int ndim = (D + 7) / 8 * 8;
    for (int d = lane; d < ndim; d += 32) {
        float a = 0.f, b = 0.f;
        if (on && d < D) {
            const float s = __ldg(sd + d);
            double bd = (double)__ldg(w2 + (size_t)k * D + d) / ((double)s * (double)s);
            if (capped) bd = fmin(bd, screen_cap(D));
            const double nu = ((double)__ldg(mu + (size_t)k * D + d) - (double)__ldg(gd + d)) * (double)s;
            a = (float)(2.0 * bd * nu / (double)q.x);
            b = (float)(-bd / (double)q.x);
        }
        const int cx = 16 * (d >> 3) + (d & 7);
        __half* o = p + ((size_t)(cx >> 6) * Kpad + pos) * 64 + (cx & 63);
        o[0] = __float2half_rn(a);
        o[8] = __float2half_rn(b);
    }
    if (lane == 0) {
        comp_of[pos] = on ? k : -1;
        float* tf = reinterpret_cast<float*>(tab) + (size_t)(pos >> 1) * 4 + (pos & 1);
        tf[0] = q.x;
        tf[2] = q.y;
        // the largest allowances of the block of 32 positions (non-negative floats order as integers), and whether it holds a
        // capped component (then it has no lower bound)
        int* bk = reinterpret_cast<int*>(blk + (pos >> 5));
        atomicMax(bk, __float_as_int(q.z));
        atomicMax(bk + 1, __float_as_int(q.w));
        if (capped) bk[2] = 1;
    }
}

// ------------------------------------------------------------------------------------------------------------------
// X -> fp16 plane [u | u^2], k-step interleaved (8 dimensions of u, the same 8 of u^2), atom by atom, and |u|^2.  L lanes per
// row, 8 dimensions each.  Bound by memory: 4 D bytes in, 4 D out.
template <int L>
__global__ void __launch_bounds__(256) screen_transform_kernel(const float* __restrict__ X, int64_t n, int D, const float* __restrict__ sd,
                                                               const float* __restrict__ gd, unsigned char* __restrict__ y,
                                                               float* __restrict__ n2, int* __restrict__ ctl, int* __restrict__ status) {
    if (blockIdx.x == 0 && threadIdx.x < 3) ctl[SC_MARKS + threadIdx.x] = 0;
    if (ctl[SC_DENSE] != 0) return;
    const bool vec_ok = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    const int l = threadIdx.x % L, d0 = l * 8;
    constexpr int RPB = 256 / L;
    float gv[8], sv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { gv[j] = __ldg(gd + d0 + j); sv[j] = __ldg(sd + d0 + j); }
    bool bad = false;
    const int64_t step = (int64_t)gridDim.x * RPB;
    auto load = [&](int64_t row, float (&x)[8]) {
        if (row < n && vec_ok && d0 + 8 <= D) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(X + row * D + d0)), b = __ldg(reinterpret_cast<const float4*>(X + row * D + d0) + 1);
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = (row < n && d0 + j < D) ? __ldg(X + row * D + d0 + j) : 0.f;
        }
    };
    auto store = [&](int64_t row, const float (&x)[8]) {
        float nrm = 0.f;
        bool far = false;
        uint32_t xh[4], qh[4];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            bad |= !(fabsf(x[j]) <= 3.0e38f) || !(fabsf(x[j + 1]) <= 3.0e38f);
            float u0 = d0 + j < D ? (x[j] - gv[j]) * sv[j] : 0.f, u1 = d0 + j + 1 < D ? (x[j + 1] - gv[j + 1]) * sv[j + 1] : 0.f;
            far |= !(fabsf(u0) <= 240.f) || !(fabsf(u1) <= 240.f);
            u0 = fminf(fmaxf(u0, -240.f), 240.f);
            u1 = fminf(fmaxf(u1, -240.f), 240.f);
            const float q0 = u0 * u0, q1 = u1 * u1;
            nrm += q0 + q1;
            const __half2 h = __floats2half2_rn(u0, u1), sq = __floats2half2_rn(q0, q1);
            xh[j / 2] = *reinterpret_cast<const uint32_t*>(&h);
            qh[j / 2] = *reinterpret_cast<const uint32_t*>(&sq);
        }
        if (far) nrm = CUDART_INF_F;                 // (a clamped coordinate: no bound holds, the row is evaluated in full)
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        if (row >= n) return;
        if (d0 < D) {
            uint4* o = reinterpret_cast<uint4*>(y + ((size_t)(l >> 2) * SCR_PIECE + row) * 128 + (l & 3) * 32);
            o[0] = make_uint4(xh[0], xh[1], xh[2], xh[3]);
            o[1] = make_uint4(qh[0], qh[1], qh[2], qh[3]);
        }
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
    if (bad) atomicOr(status, ST_BAD_X);
}

// ------------------------------------------------------------------------------------------------------------------
// Sweep
constexpr int SW_THREADS = 320;              // 8 softmax warps, producer warp, MMA warp
constexpr int SW_PRODUCER = 8, SW_MMA = 9;
constexpr int SW_YSLOT = 32768, SW_YS = 4;   // atoms of 256 points
constexpr int SW_PSLOT = 16384, SW_PS = 4;   // atoms of 128 components
constexpr int SW_ENT = 14;                   // groups of 32 components a point can have marks in
constexpr int SW_POFF = SW_YS * SW_YSLOT;
constexpr int SW_EOFF = SW_POFF + SW_PS * SW_PSLOT;
constexpr int SW_TOFF = SW_EOFF + SW_ENT * 256 * 8;      // tables: 2 x (64 float4 + 4 float2)
constexpr int SW_BOFF = SW_TOFF + 2 * 1088;
constexpr int SW_SMEM = SW_BOFF + 256 + 1024;
enum { SB_PFULL = 0, SB_PEMPTY = SB_PFULL + SW_PS, SB_YFULL = SB_PEMPTY + SW_PS, SB_YEMPTY = SB_YFULL + SW_YS, SB_LFULL = SB_YEMPTY + SW_YS,
       SB_LEMPTY = SB_LFULL + 2, SB_FINAL = SB_LEMPTY + 2, SB_COUNT };
static_assert(SB_COUNT * 8 <= 256, "barriers");
static_assert(SW_SMEM <= 232448, "shared memory");

// two fp32 operations per instruction
__device__ __forceinline__ uint64_t pack2(uint32_t a, uint32_t b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ float lo2(uint64_t a) { return __uint_as_float((uint32_t)a); }
__device__ __forceinline__ float hi2(uint64_t a) { return __uint_as_float((uint32_t)(a >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
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
    float margin;
    const float4* tab;
    const int4* blk;
    const int* comp_of;
    const float* n2;
    unsigned* pt_off;
    int* pt_cnt;
    unsigned short* ids;
    int* ovf;
    int* ctl;
    int* status;
};

// Tile = 256 points, two MMAs of M = 128 per coefficient atom: a tile of 128 would need the coefficients twice as often (64
// bytes per cycle and SM at D = 128, about what L2 delivers).  An accumulator buffer is 128 components x 2 halves of the tile;
// two buffers alternate, so the softmax warps read one group while the tensor cores form the next.  MMA time per group of 128
// components: 2 x ceil(D / 8) x 64.5 cycles; softmax: about 170 instructions per 32 values.
__global__ void __launch_bounds__(SW_THREADS, 1)
screen_sweep_kernel(const SweepParams p, const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, drain_s;
    if (p.ctl[SC_DENSE] != 0) return;
    volatile int* abort_flag = &abort_s;
    volatile int* drain_flag = &drain_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t ntiles = (p.n + SCR_TILE - 1) / SCR_TILE;
    const int64_t ntl = ((int64_t)blockIdx.x < ntiles) ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    const int KA = p.KA, NG = p.NG;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SW_BOFF);
    auto BAR = [&](int i) { return smem_u32(&bars[i]); };
    if (tid == 0) {
        abort_s = 0;
        drain_s = 0;
        for (int i = 0; i < SB_COUNT; ++i) bar_init(BAR(i), (i == SB_LEMPTY || i == SB_LEMPTY + 1) ? 256 : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == SW_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_base_s;

    if (warp < 8) {
        // =========================== softmax warps: thread = TMEM lane = point ===========================
        const int half = warp >> 2;
        const uint32_t lane_addr = ((uint32_t)((warp & 3) * 32)) << 16;
        unsigned long long* ent = reinterpret_cast<unsigned long long*>(smem + SW_EOFF) + tid;        // entry e at ent[256 e]
        uint32_t gi = 0;                                     // groups processed (all tiles)
        int marks = 0;
        float4 nt = make_float4(0.f, 0.f, 0.f, 0.f);
        float2 nb = make_float2(0.f, 0.f);
        auto table_load = [&](int g) {
            if (tid < 64) nt = __ldg(p.tab + g * 64 + tid);
            else if (tid < 68) {
                const int4 q = __ldg(p.blk + g * 4 + tid - 64);
                nb = make_float2(q.z ? -__int_as_float(q.x) : __int_as_float(q.x), __int_as_float(q.y));      // (sign: no lower bound)
            }
        };
        auto table_store = [&](uint32_t b) {
            unsigned char* t = smem + SW_TOFF + b * 1088;
            if (tid < 64) reinterpret_cast<float4*>(t)[tid] = nt;
            else if (tid < 68) reinterpret_cast<float2*>(t + 1024)[tid - 64] = nb;
        };
        for (int64_t i = 0; i < ntl; ++i) {
            const int64_t wrow = (blockIdx.x + i * gridDim.x) * SCR_TILE + warp * 32;       // first row of this warp
            const int64_t row = wrow + lane;
            const bool in = row < p.n;
            const float nrm = in ? __ldg(p.n2 + row) : 0.f;
            float thr = -CUDART_INF_F;                       // the largest lower bound so far
            int ne = 0;
            float lost = -CUDART_INF_F;                      // largest upper bound of a block with marks that found no room
            // 32 accumulators of the point: approximate values l = t acc + c, two at a time; the block's largest; marks.
            auto block = [&](const uint32_t (&v)[32], int bn, const float4* t4, float2 ab) {
                uint64_t l[16];
                float mx[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(t4 + j);      // same address in every lane
                    l[j] = fma2(pack2(v[2 * j], v[2 * j + 1]), t.x, t.y);
                    mx[j & 3] = max3(mx[j & 3], lo2(l[j]), hi2(l[j]));
                }
                const float bmax = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]), E = fmaf(ab.y, nrm, fabsf(ab.x));
                if (!(ab.x < 0.f)) thr = fmaxf(thr, bmax - E);
                const float cut = thr - p.margin - E;
                if (in && bmax >= cut && bmax > -CUDART_INF_F) {
                    // bit j of the mask: value j reaches the cut (the sign of l - cut, shifted in from the top)
                    const uint64_t nc = pack2(__float_as_uint(-cut), __float_as_uint(-cut));
                    unsigned mask = 0;
#pragma unroll
                    for (int j = 15; j >= 0; --j) {
                        const uint64_t d = add2(l[j], nc);
                        mask = __funnelshift_l(__float_as_uint(hi2(d)), mask, 1);
                        mask = __funnelshift_l(__float_as_uint(lo2(d)), mask, 1);
                    }
                    mask = ~mask;
                    if (ne == SW_ENT) {                      // drop what the bound found meanwhile rules out
                        int m = 0;
                        for (int e = 0; e < SW_ENT; ++e) {
                            const unsigned long long w = ent[256 * e];
                            if (__uint_as_float((unsigned)(w >> 32) & ~255u) >= thr - p.margin) ent[256 * m++] = w;
                        }
                        ne = m;
                    }
                    const float ub = bmax + E;
                    if (ne < SW_ENT) {
                        // the block's largest upper bound, rounded up to the 24 bits that share a word with its number
                        const unsigned ubits = (__float_as_uint(ub + fabsf(ub) * 1e-4f + 1e-3f) & ~255u) | (unsigned)bn;
                        ent[256 * ne++] = ((unsigned long long)ubits << 32) | mask;
                    } else {
                        lost = fmaxf(lost, ub);              // (harmless if the final bound rules the block out)
                    }
                }
            };
            table_load(0);
            table_store(gi & 1);
            for (int g = 0; g < NG; ++g, ++gi) {
                const uint32_t buf = gi & 1;
                named_bar_sync(1, 256);                      // the group's table is in place, the other one free
                if (g + 1 < NG) table_load(g + 1);
                const bool got = bar_wait(BAR(SB_LFULL + buf), (gi >> 1) & 1u, abort_flag, p.status, false);
                const bool ok = __all_sync(0xffffffffu, got);
                fence_after();
                const float4* tab = reinterpret_cast<const float4*>(smem + SW_TOFF + buf * 1088);
                const float2* blk = reinterpret_cast<const float2*>(smem + SW_TOFF + buf * 1088 + 1024);
                if (ok) {
                    const uint32_t col = tmem + buf * 256 + half * 128 + lane_addr;
                    uint32_t va[32], vb[32];
                    tmem_ld32(col, va);
                    tmem_wait(va);
                    tmem_ld32(col + 32, vb);
                    block(va, g * 4, tab, blk[0]);
                    tmem_wait(vb);
                    tmem_ld32(col + 64, va);
                    block(vb, g * 4 + 1, tab + 16, blk[1]);
                    tmem_wait(va);
                    tmem_ld32(col + 96, vb);
                    block(va, g * 4 + 2, tab + 32, blk[2]);
                    tmem_wait(vb);
                    block(vb, g * 4 + 3, tab + 48, blk[3]);
                }
                fence_before();
                bar_arrive(BAR(SB_LEMPTY + buf));
                if (g + 1 < NG) table_store(buf ^ 1);
            }
            // the point's list: what the final bound leaves
            int cnt = 0;
            const float fin = thr - p.margin;
            bool over = !(nrm < CUDART_INF_F) || lost >= fin && lost > -CUDART_INF_F;
            if (in && !over)
                for (int e = 0; e < ne; ++e) {
                    const unsigned long long w = ent[256 * e];
                    if (__uint_as_float((unsigned)(w >> 32) & ~255u) >= fin) cnt += __popc((unsigned)w);
                }
            int inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if (inc > 32 * SCR_SLOTS) over = true;
            if (in && !*abort_flag) {
                unsigned o = (unsigned)(wrow * SCR_SLOTS) + (unsigned)(inc - cnt);
                p.pt_off[row] = o;
                p.pt_cnt[row] = over ? 0 : cnt;
                if (over) {
                    p.ovf[atomicAdd(p.ctl + SC_OVF, 1)] = (int)row;
                } else {
                    marks += cnt;
                    for (int e = 0; e < ne; ++e) {
                        const unsigned long long w = ent[256 * e];
                        if (!(__uint_as_float((unsigned)(w >> 32) & ~255u) >= fin)) continue;
                        unsigned mask = (unsigned)w;
                        const int base = (int)((w >> 32) & 255u) * 32;
                        while (mask) {
                            const int j = __ffs(mask) - 1;
                            mask &= mask - 1;
                            p.ids[o++] = (unsigned short)__ldg(p.comp_of + base + j);
                        }
                    }
                }
            }
            named_bar_sync(2, 256);                          // (the tables are rewritten by the next tile)
        }
        marks = __reduce_add_sync(0xffffffffu, marks);
        if (lane == 0 && marks > 0) atomicAdd(p.ctl + SC_MARKS, marks);
    } else if (warp == SW_PRODUCER) {
        // =========================== producer warp (TMA) ===========================
        uint32_t ps = 0, ya = 0;                             // stages and atoms requested so far
        bool ok = true;
        const uint64_t keep = l2_policy_evict_last();
        auto wait_slot = [&](int bar, uint32_t parity) -> bool {
            uint32_t w = 1;
            if (lane == 0) w = bar_wait(BAR(bar), parity, abort_flag, p.status, false) ? 1u : 0u;
            return __shfl_sync(0xffffffffu, w, 0) != 0u;
        };
        for (int64_t i = 0; i < ntl && ok; ++i) {
            const int32_t row0 = (int32_t)((blockIdx.x + i * gridDim.x) * SCR_TILE);
            for (int g = 0; g < NG && ok; ++g)
                for (int z = 0; z < KA && ok; ++z) {
                    if (g == 0) {
                        const uint32_t slot = ya % SW_YS;
                        if (ya >= SW_YS) ok = wait_slot(SB_YEMPTY + slot, (ya / SW_YS - 1) & 1u);
                        if (!ok) break;
                        if (elect_one()) {
                            bar_expect_tx(BAR(SB_YFULL + slot), SW_YSLOT);
                            tma_load_3d(smem_u32(smem + slot * SW_YSLOT), &tm_y, 0, row0, z, BAR(SB_YFULL + slot));
                        }
                        __syncwarp();
                        ++ya;
                    }
                    const uint32_t slot = ps % SW_PS;
                    if (ps >= SW_PS) ok = wait_slot(SB_PEMPTY + slot, (ps / SW_PS - 1) & 1u);
                    if (!ok) break;
                    if (elect_one()) {
                        bar_expect_tx(BAR(SB_PFULL + slot), SW_PSLOT);
                        tma_load_3d_hint(smem_u32(smem + SW_POFF + slot * SW_PSLOT), &tm_p, 0, g * 128, z, BAR(SB_PFULL + slot), keep);
                        // the next tile's atoms into L2 while this one is worked on
                        if (g == 0 && i + 1 < ntl) tma_prefetch_3d(&tm_y, 0, (int32_t)(row0 + (int64_t)gridDim.x * SCR_TILE), z);
                    }
                    __syncwarp();
                    ++ps;
                }
        }
        // the loads in flight must have landed before the CTA may exit, also after an abort
        if (!ok || *abort_flag) {
            for (uint32_t h = (ps > SW_PS ? ps - SW_PS : 0); h < ps; ++h) {
                if (lane == 0) bar_wait(BAR(SB_PFULL + h % SW_PS), (h / SW_PS) & 1u, drain_flag, p.status, false);
                __syncwarp();
            }
            for (uint32_t h = (ya > SW_YS ? ya - SW_YS : 0); h < ya; ++h) {
                if (lane == 0) bar_wait(BAR(SB_YFULL + h % SW_YS), (h / SW_YS) & 1u, drain_flag, p.status, false);
                __syncwarp();
            }
        }
    } else {
        // =========================== MMA warp ===========================
        const uint32_t idesc = make_idesc(128, 128, 0);
        const uint64_t dy = make_desc(smem_u32(smem), 16, 1024), dp = make_desc(smem_u32(smem + SW_POFF), 16, 1024);
        auto wait_all = [&](int bar, uint32_t parity) -> bool {
            uint32_t ok = 1;
            if (lane == 0) ok = bar_wait(BAR(bar), parity, abort_flag, p.status, false) ? 1u : 0u;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            fence_after();
            return ok != 0u;
        };
        uint32_t ps = 0, ya = 0, gi = 0;
        bool alive = true;
        for (int64_t i = 0; i < ntl && alive; ++i) {
            for (int g = 0; g < NG && alive; ++g, ++gi) {
                const uint32_t buf = gi & 1;
                if (gi >= 2 && !wait_all(SB_LEMPTY + buf, (gi / 2 - 1) & 1u)) { alive = false; break; }
                const uint32_t d = tmem + buf * 256;
                for (int z = 0; z < KA; ++z) {
                    const uint32_t yslot = (ya + z) % SW_YS, slot = ps % SW_PS;
                    if (g == 0 && !wait_all(SB_YFULL + yslot, ((ya + z) / SW_YS) & 1u)) { alive = false; break; }
                    if (!wait_all(SB_PFULL + slot, (ps / SW_PS) & 1u)) { alive = false; break; }
                    ++ps;
                    const int nk = (p.KS - 4 * z < 4) ? (p.KS - 4 * z) : 4;
                    if (elect_one()) {
                        const uint64_t a = dy + ((yslot * SW_YSLOT) >> 4), b = dp + ((slot * SW_PSLOT) >> 4);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (j < nk) {
                                const uint32_t acc = (z > 0 || j > 0) ? 1u : 0u;
                                mma_ss(d, a + ((j * 32) >> 4), b + ((j * 32) >> 4), idesc, acc);
                                mma_ss(d + 128, a + ((16384 + j * 32) >> 4), b + ((j * 32) >> 4), idesc, acc);
                            }
                        mma_commit(BAR(SB_PEMPTY + slot));
                        if (g == NG - 1) mma_commit(BAR(SB_YEMPTY + yslot));
                        if (z == KA - 1) mma_commit(BAR(SB_LFULL + buf));
                    }
                    __syncwarp();
                }
            }
            ya += KA;
        }
        if (elect_one()) mma_commit(BAR(SB_FINAL));
        __syncwarp();
        if (lane == 0) bar_wait(BAR(SB_FINAL), 0, drain_flag, p.status, false);
        __syncwarp();
        fence_after();
    }
    fence_before();
    __syncthreads();
    if (warp == SW_MMA) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------------------------
// Rows that left the sweep without a list (marks in too many groups of components, a coordinate beyond the fp16 range): all K
// components exactly, the list from those values.  Four rows per CTA and step, a warp per component.  Also the verdict on the
// piece: with too many such rows, or too many pairs, SC_DENSE is set and nothing after this kernel does anything.
constexpr int OV_ROWS = 4;
__global__ void __launch_bounds__(256) screen_rows_kernel(const float* __restrict__ X, int64_t n, int D, int K, float margin,
                                                          long long max_marks, const float* __restrict__ mu, const float* __restrict__ w2,
                                                          const double* __restrict__ c2d, const int* __restrict__ ovf,
                                                          unsigned* __restrict__ pt_off, int* __restrict__ pt_cnt,
                                                          unsigned short* __restrict__ ids, int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
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
            const float cut = best - margin - 0.01f;
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
// Exact values.  A warp takes 32 points: their listed pairs (of the points that have more than one) go into a work list in
// shared memory, four pairs are evaluated at a time, eight lanes each - a lane holds every eighth group of four dimensions -
// and then a lane per point reads its values back.  (Eight lanes per POINT took the time of the longest of four lists.)
// Bound by instruction issue and the trips to L2 for the components' rows (1 KB per pair at D = 128).
constexpr int EV_VALS = 32 * SCR_SLOTS;
template <int MODE>
__global__ void __launch_bounds__(256, 3) screen_eval_kernel(const float* __restrict__ X, int64_t n, int D, int K, const float* __restrict__ mu,
                                                             const float* __restrict__ w2, const double* __restrict__ c2d,
                                                             const unsigned* __restrict__ pt_off, int* __restrict__ pt_cnt,
                                                             unsigned short* __restrict__ ids, float* __restrict__ val,
                                                             int* __restrict__ counts, double* __restrict__ ll, float* __restrict__ logp,
                                                             int32_t* __restrict__ idx, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    extern __shared__ int hist[];                    // [K] (unless MODE == SCREEN_LOGP)
    __shared__ float v_s[8][EV_VALS];                // values of the warp's pairs, by position in its part of the lists
    __shared__ unsigned short w_s[8][EV_VALS];       // work list: point (5 bits), position (9 bits)
    __shared__ double red[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l8 = lane & 7;
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0) && ((reinterpret_cast<uintptr_t>(mu) & 15) == 0);
    const bool histogram = MODE != SCREEN_LOGP && counts != nullptr;
    if (histogram) {
        for (int k = tid; k < K; k += 256) hist[k] = 0;
        __syncthreads();
    }
    // c - sum_d w (x - m)^2, the same in the eight lanes that call together; dimensions 4 (l8 + 8 i) + (0..3)
    auto pair_value = [&](const float* __restrict__ x, int k) -> float {
        const float *m = mu + (size_t)k * D, *w = w2 + (size_t)k * D;
        float q = 0.f;
        if (vec) {
            float4 a[4], b[4], c[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int d = 4 * (l8 + 8 * i);
                a[i] = b[i] = c[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (d < D) {
                    a[i] = __ldg(reinterpret_cast<const float4*>(x + d));
                    b[i] = __ldg(reinterpret_cast<const float4*>(m + d));
                    c[i] = __ldg(reinterpret_cast<const float4*>(w + d));
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float t0 = a[i].x - b[i].x, t1 = a[i].y - b[i].y, t2 = a[i].z - b[i].z, t3 = a[i].w - b[i].w;
                q = fmaf(c[i].x * t0, t0, q); q = fmaf(c[i].y * t1, t1, q); q = fmaf(c[i].z * t2, t2, q); q = fmaf(c[i].w * t3, t3, q);
            }
        } else {
            for (int d = l8; d < D; d += 8) { const float t = __ldg(x + d) - __ldg(m + d); q = fmaf(__ldg(w + d) * t, t, q); }
        }
        q += __shfl_xor_sync(0xffffffffu, q, 1);
        q += __shfl_xor_sync(0xffffffffu, q, 2);
        q += __shfl_xor_sync(0xffffffffu, q, 4);
        return (float)(__ldg(c2d + k) - (double)q);
    };
    double ll_acc = 0.0;
    for (int it = 0; it < SCR_RANGE / 256; ++it) {
        const int64_t row0 = (int64_t)blockIdx.x * SCR_RANGE + it * 256 + warp * 32, row = row0 + lane;
        if (row0 >= n) break;
        const bool in = row < n;
        const int cnt = in ? pt_cnt[row] : 0;
        const unsigned off = in ? pt_off[row] : 0u, base = (unsigned)(row0 * SCR_SLOTS);
        const bool listed = off < (unsigned)(SCR_PIECE * SCR_SLOTS);             // (else: a row with a list of its own length)
        const bool alone = cnt == 1 && MODE != SCREEN_LOGP;                      // its value is not needed here
        const int todo = (!listed || alone) ? 0 : cnt;
        int inc = todo;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        const int total = __shfl_sync(0xffffffffu, inc, 31), p0 = (int)(off - base);
        __syncwarp();
        for (int j = 0; j < todo; ++j) w_s[warp][inc - todo + j] = (unsigned short)((lane << 9) | (p0 + j));
        __syncwarp();
        for (int s = 0; s < total; s += 4) {
            const int item = s + (lane >> 3);
            const int w = w_s[warp][min(item, total - 1)];
            const int k = ids[base + (w & 511)];
            const float l = pair_value(X + (row0 + (w >> 9)) * D, k);
            if (l8 == 0 && item < total) v_s[warp][w & 511] = l;
        }
        __syncwarp();
        float mx = -CUDART_INF_F, sum = 0.f;
        int best = 0, kept = 0;
        if (listed && cnt > 0) {
            if (MODE == SCREEN_ARGMAX) {
                best = ids[off];
                if (!alone) {
                    mx = v_s[warp][p0];
                    for (int j = 1; j < cnt; ++j) {
                        const float l = v_s[warp][p0 + j];
                        const int k = ids[off + j];
                        if (l > mx || (l == mx && k < best)) { mx = l; best = k; }
                    }
                }
            } else if (!alone) {
                for (int j = 0; j < cnt; ++j) mx = fmaxf(mx, v_s[warp][p0 + j]);
                for (int j = 0; j < cnt; ++j) sum += fast_ex2(v_s[warp][p0 + j] - mx);
            }
        }
        // rows with lists of their own length: the whole warp, one row after the other, values in `val`
        for (unsigned todo_rows = __ballot_sync(0xffffffffu, in && !listed); todo_rows;) {
            const int src = __ffs(todo_rows) - 1;
            todo_rows &= todo_rows - 1;
            const int c = __shfl_sync(0xffffffffu, cnt, src);
            const unsigned o = __shfl_sync(0xffffffffu, off, src);
            float m = -CUDART_INF_F, sm = 0.f;
            int b = 0;
            for (int s = 0; s < c; s += 4) {
                const int j = min(s + (lane >> 3), c - 1);
                const int k = ids[o + j];
                const float l = pair_value(X + (row0 + src) * D, k);
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
            const float lz = m + log2f(sm);
            int kp = 0;
            if (MODE == SCREEN_EM)
                for (int j0 = 0; j0 < c; j0 += 32) {
                    const int j = j0 + lane;
                    const float r = j < c ? fast_ex2(val[o + j] - lz) : 0.f;
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
        if (MODE == SCREEN_LOGP) {
            if (in) {
                const double lz = cnt > 0 ? (double)mx + (double)log2f(sum) : -CUDART_INF;
                logp[row] = (float)(lz * 0.69314718055994530942);
                ll_acc += lz;
            }
        } else if (MODE == SCREEN_ARGMAX) {
            if (in) {
                if (idx) idx[row] = best;
                if (histogram && cnt > 0) {
                    ids[off] = (unsigned short)best;
                    val[off] = -1.f;
                    pt_cnt[row] = 1;
                    atomicAdd(&hist[best], 1);
                }
            }
        } else if (in) {
            // responsibilities; the pairs below 2^-40 of the total leave the list
            if (cnt == 0) {
                ll_acc += -CUDART_INF;
            } else if (listed && alone) {
                val[off] = -1.f;
                atomicAdd(&hist[ids[off]], 1);
            } else {
                ll_acc += (double)mx + (double)log2f(sum);
                if (listed) {
                    const float lz = mx + log2f(sum);
                    for (int j = 0; j < cnt; ++j) {
                        const float r = fast_ex2(v_s[warp][p0 + j] - lz);
                        if (r >= 9.094947e-13f) {
                            const unsigned short id = ids[off + j];
                            ids[off + kept] = id;
                            val[off + kept] = r;
                            ++kept;
                            atomicAdd(&hist[id], 1);
                        }
                    }
                }
                pt_cnt[row] = kept;
            }
        }
        __syncwarp();
    }
    if (histogram) {
        __syncthreads();
        for (int k = tid; k < K; k += 256) counts[(size_t)blockIdx.x * K + k] = hist[k];
    }
    if (MODE != SCREEN_ARGMAX && ll) {
        ll_acc = warp_sum(ll_acc);
        if (lane == 0) red[warp] = ll_acc;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += red[w];
            ll[blockIdx.x] += s * 0.69314718055994530942;            // one owner per slot: launches add up
        }
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

// A CTA per range, a warp per 64 points of it, with cursors of its own: lanes = points, their pairs one after the other, the
// pairs of one component ranked by lane.  The order is the same in every run.
__global__ void __launch_bounds__(256) screen_fill_kernel(int64_t n, int K, const unsigned* __restrict__ pt_off, const int* __restrict__ pt_cnt,
                                                          const unsigned short* __restrict__ ids, const float* __restrict__ val,
                                                          const int* __restrict__ starts, const int* __restrict__ off,
                                                          uint2* __restrict__ srt, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    extern __shared__ int sm[];                      // base [K], then the warps' cursors [8][K rounded up to even] as 16-bit values
    const int K2 = (K + 1) & ~1;
    int* base = sm;
    unsigned* cur32 = reinterpret_cast<unsigned*>(sm + K2);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned short* cur = reinterpret_cast<unsigned short*>(cur32) + (size_t)warp * K2;
    for (int k = tid; k < K; k += 256) base[k] = __ldg(off + k) + starts[(size_t)blockIdx.x * K + k];
    for (int k = tid; k < 4 * K2; k += 256) cur32[k] = 0u;
    __syncthreads();
    const int64_t p0 = (int64_t)blockIdx.x * SCR_RANGE + warp * (SCR_RANGE / 8);
    int cnt[2];
    unsigned o[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t row = p0 + 32 * h + lane;
        cnt[h] = row < n ? pt_cnt[row] : 0;
        o[h] = row < n ? pt_off[row] : 0u;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        for (int j = 0; j < cnt[h]; ++j) {
            const int k = ids[o[h] + j];
            atomicAdd(cur32 + ((size_t)warp * K2 + k) / 2, 1u << (16 * (k & 1)));
        }
    __syncthreads();
    for (int k = tid; k < K; k += 256) {
        unsigned c = 0;
        unsigned short* q = reinterpret_cast<unsigned short*>(cur32) + k;
#pragma unroll
        for (int w = 0; w < 8; ++w) { const unsigned v = q[(size_t)w * K2]; q[(size_t)w * K2] = (unsigned short)c; c += v; }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int most = __reduce_max_sync(0xffffffffu, (unsigned)cnt[h]);
        for (int j = 0; j < most; ++j) {
            const bool on = j < cnt[h];
            const int k = on ? ids[o[h] + j] : -1;
            const float r = on ? val[o[h] + j] : 0.f;
            const unsigned peers = __match_any_sync(0xffffffffu, k);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            int c = 0;
            if (on) c = cur[k];
            __syncwarp();
            if (on) {
                if (rank == 0) cur[k] = (unsigned short)(c + __popc(peers));
                srt[base[k] + c + rank] = make_uint2((unsigned)(p0 + 32 * h + lane), __float_as_uint(r));
            }
            __syncwarp();
        }
    }
}

// Statistics of one work item (at most SCR_SEG pairs of one component) by one warp: sums of r, r (x - mu), r (x - mu)^2 in
// fp32, and, over the points whose only pair this is, their number and sum_d w2 (x - mu)^2 (their log-likelihood).  lpr lanes
// per row, four dimensions each; the rows of four steps are in flight together.
__global__ void __launch_bounds__(256) screen_stats_kernel(const float* __restrict__ X, int D, int lpr, const float* __restrict__ mu,
                                                           const float* __restrict__ w2, const uint2* __restrict__ srt,
                                                           const int* __restrict__ off, const int* __restrict__ segoff,
                                                           int K, float* __restrict__ part, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    extern __shared__ int seg_s[];                   // [K + 1]
    for (int j = threadIdx.x; j <= K; j += 256) seg_s[j] = segoff[j];
    __syncthreads();
    const int lane = threadIdx.x & 31, l = lane % lpr, sub = lane / lpr, rows = 32 / lpr;
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
    const int items = seg_s[K], nw = gridDim.x * 8;
    const int d0 = 4 * l;
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
    for (int item = blockIdx.x * 8 + (threadIdx.x >> 5); item < items; item += nw) {
        int k = 0;                                   // the component whose items hold this one: the last with segoff <= item
        for (int w = K; w > 1;) {
            const int h = w >> 1;
            if (seg_s[k + h] <= item) k += h;
            w -= h;
        }
        const int a = __ldg(off + k) + (item - seg_s[k]) * SCR_SEG, b = min(a + SCR_SEG, __ldg(off + k + 1));
        const float4 m = load4(mu + (size_t)k * D, false), w = load4(w2 + (size_t)k * D, false);
        float4 s1 = make_float4(0.f, 0.f, 0.f, 0.f), s2 = s1;
        float nsum = 0.f, n1 = 0.f, q1 = 0.f;
        for (int p = a; p < b; p += 32) {
            uint2 e = make_uint2(0u, 0u);
            if (p + lane < b) e = __ldg(srt + p + lane);
            const float re = __uint_as_float(e.y);
            nsum += fabsf(re);
            n1 += re < 0.f ? 1.f : 0.f;
            const int have = min(32, b - p);
            for (int i = 0; i < have; i += 4 * rows) {
                float4 x[4];
                float r[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int src = min(31, i + u * rows + sub);
                    const unsigned row = __shfl_sync(0xffffffffu, e.x, src);
                    r[u] = __shfl_sync(0xffffffffu, re, src);
                    if (i + u * rows + sub >= have) r[u] = 0.f;
                    x[u] = make_float4(m.x, m.y, m.z, m.w);
                    if (r[u] != 0.f) x[u] = load4(X + (size_t)row * D, vec);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float ra = fabsf(r[u]);
                    const float tx = x[u].x - m.x, ty = x[u].y - m.y, tz = x[u].z - m.z, tw = x[u].w - m.w;
                    s1.x = fmaf(ra, tx, s1.x); s1.y = fmaf(ra, ty, s1.y); s1.z = fmaf(ra, tz, s1.z); s1.w = fmaf(ra, tw, s1.w);
                    const float ax = tx * tx, ay = ty * ty, az = tz * tz, aw = tw * tw;
                    s2.x = fmaf(ra, ax, s2.x); s2.y = fmaf(ra, ay, s2.y); s2.z = fmaf(ra, az, s2.z); s2.w = fmaf(ra, aw, s2.w);
                    const float q = fmaf(w.x, ax, fmaf(w.y, ay, fmaf(w.z, az, w.w * aw)));
                    if (r[u] < 0.f) q1 += q;
                }
            }
        }
        for (int o = lpr; o < 32; o <<= 1) {
            s1.x += __shfl_xor_sync(0xffffffffu, s1.x, o); s1.y += __shfl_xor_sync(0xffffffffu, s1.y, o);
            s1.z += __shfl_xor_sync(0xffffffffu, s1.z, o); s1.w += __shfl_xor_sync(0xffffffffu, s1.w, o);
            s2.x += __shfl_xor_sync(0xffffffffu, s2.x, o); s2.y += __shfl_xor_sync(0xffffffffu, s2.y, o);
            s2.z += __shfl_xor_sync(0xffffffffu, s2.z, o); s2.w += __shfl_xor_sync(0xffffffffu, s2.w, o);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            nsum += __shfl_xor_sync(0xffffffffu, nsum, o);
            n1 += __shfl_xor_sync(0xffffffffu, n1, o);
            q1 += __shfl_xor_sync(0xffffffffu, q1, o);
        }
        float* po = part + (size_t)item * (2 * D + 3);
        if (sub == 0) {
            const float v1[4] = {s1.x, s1.y, s1.z, s1.w}, v2[4] = {s2.x, s2.y, s2.z, s2.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (d0 + j < D) { po[d0 + j] = v1[j]; po[D + d0 + j] = v2[j]; }
        }
        if (lane == 0) { po[2 * D] = nsum; po[2 * D + 1] = n1; po[2 * D + 2] = q1; }
    }
}

// A CTA per component: its items in order (eight interleaved chains, then those in order), float64, shifted from its mean to
// the origin.
__global__ void __launch_bounds__(1024) screen_reduce_kernel(int D, int K, const float* __restrict__ part, const int* __restrict__ segoff,
                                                             const float* __restrict__ mu, const double* __restrict__ c2d,
                                                             double* __restrict__ Nk, double* __restrict__ S1, double* __restrict__ S2,
                                                             double* __restrict__ llk, const int* __restrict__ ctl) {
    if (ctl[SC_DENSE] != 0) return;
    const int k = blockIdx.x, d = threadIdx.x & 127, r = threadIdx.x >> 7;
    const int i0 = segoff[k], i1 = segoff[k + 1];
    if (i0 == i1) return;
    __shared__ double sh[8][128][2];
    __shared__ double tot[3];
    const size_t st = (size_t)(2 * D + 3);
    double a = 0.0, b = 0.0;
    for (int i = i0 + r; i < i1; i += 32) {
        float qa[4], qb[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = i + 8 * u < i1 && d < D;
            const float* q = part + (size_t)(i + 8 * u) * st;
            qa[u] = in ? q[d] : 0.f;
            qb[u] = in ? q[D + d] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) { a += (double)qa[u]; b += (double)qb[u]; }
    }
    sh[r][d][0] = a;
    sh[r][d][1] = b;
    if (threadIdx.x < 96) {                              // warp q: the item's q-th scalar (weight, lone points, their quadratic forms)
        const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
        double s = 0.0;
        for (int i = i0 + lane; i < i1; i += 32) s += (double)part[(size_t)i * st + 2 * D + q];
        s = warp_sum(s);
        if (lane == 0) tot[q] = s;
    }
    __syncthreads();
    if (r != 0) return;
    const double n = tot[0];
    if (d < D) {
        a = b = 0.0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { a += sh[j][d][0]; b += sh[j][d][1]; }
        const double m = (double)__ldg(mu + (size_t)k * D + d);
        S1[(size_t)k * D + d] += a + m * n;
        S2[(size_t)k * D + d] += b + 2.0 * m * a + m * m * n;
    }
    if (d == 0) {
        Nk[k] += n;
        llk[k] += (tot[1] > 0.0 ? tot[1] * c2d[k] - tot[2] : 0.0) * 0.69314718055994530942;
    }
}

// A plane [atoms][rows][128 bytes] as a 3-D tensor: boxes of box_rows rows of one atom, 128-byte swizzle.
cudaError_t plane_map(CUtensorMap* tm, void* base, int64_t rows, int atoms, int box_rows) {
    const cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)atoms};
    const cuuint64_t strides[2] = {128, (cuuint64_t)rows * 128};
    const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    typedef CUresult (*encode_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static encode_fn encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<encode_fn>(fn);
    }
    const CUresult r = encode(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, base, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

#define LCHECK()                                       \
    do {                                               \
        const cudaError_t e_ = cudaGetLastError();     \
        if (e_ != cudaSuccess) return e_;              \
    } while (0)

}  // namespace

bool screen_supports(int D, int K) { return D >= 1 && D <= 128 && K >= 1 && K <= SCR_MAX_K; }

cudaError_t launch_screen_prepare(cudaStream_t s, int D, int K, const float* pi, const float* mu, const float* var, bool unit,
                                  const ScreenBuffers& b, float* w2, float* c2, double* c2d, int* status) {
    const int Kpad = screen_kpad(K);
    const int db = (K + 7) / 8 < SCR_DIM_BLOCKS ? (K + 7) / 8 : SCR_DIM_BLOCKS;
    screen_dim_kernel<<<db, 512, 0, s>>>(D, K, pi, mu, var, unit ? 1 : 0, b.dimpart, b.sd, b.gd, b.ctl);
    LCHECK();
    screen_comp_kernel<<<(K + 7) / 8, 256, 0, s>>>(D, K, pi, mu, var, unit ? 1 : 0, b.sd, b.gd, w2, c2, c2d, b.prm, b.key, b.blk, b.ctl, status);
    LCHECK();
    screen_plane_kernel<<<Kpad / 8, 256, 0, s>>>(D, K, Kpad, mu, w2, b.sd, b.gd, b.prm, b.key, reinterpret_cast<__half*>(b.p), b.tab,
                                                 b.blk, b.comp_of);
    return cudaGetLastError();
}

cudaError_t launch_screen_sweep(cudaStream_t s, const float* X, int64_t n, int D, int K, float margin, float max_marks,
                                const float* mu, const float* w2, const double* c2d, const ScreenBuffers& b, int* status, int sms,
                                int64_t* launches) {
    if (n < 1 || n > SCR_PIECE) return cudaErrorInvalidValue;
    const int KS = (D + 7) / 8;
    int64_t blocks;
    {
        int L = 1;
        while (L < KS) L <<= 1;
        const int rpb = 256 / L;
        blocks = (n + 2 * rpb - 1) / (2 * rpb);
        if (blocks > (int64_t)sms * 8) blocks = (int64_t)sms * 8;
#define FG_TR(L_) screen_transform_kernel<L_><<<(unsigned)blocks, 256, 0, s>>>(X, n, D, b.sd, b.gd, b.y, b.n2, b.ctl, status)
        switch (L) {
            case 1: FG_TR(1); break;
            case 2: FG_TR(2); break;
            case 4: FG_TR(4); break;
            case 8: FG_TR(8); break;
            default: FG_TR(16); break;
        }
#undef FG_TR
        LCHECK();
    }
    CUtensorMap my, mp;
    const int Kpad = screen_kpad(K), KA = screen_atoms(D);
    cudaError_t e = plane_map(&my, b.y, SCR_PIECE, KA, SCR_TILE);
    if (e != cudaSuccess) return e;
    e = plane_map(&mp, b.p, Kpad, KA, 128);
    if (e != cudaSuccess) return e;
    SweepParams p;
    p.n = n; p.KA = KA; p.KS = KS; p.NG = Kpad / 128; p.margin = margin;
    p.tab = b.tab; p.blk = b.blk; p.comp_of = b.comp_of; p.n2 = b.n2; p.pt_off = b.pt_off; p.pt_cnt = b.pt_cnt; p.ids = b.ids;
    p.ovf = b.ovf; p.ctl = b.ctl; p.status = status;
    e = cudaFuncSetAttribute(screen_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SW_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + SCR_TILE - 1) / SCR_TILE;
    screen_sweep_kernel<<<(unsigned)(tiles < sms ? tiles : sms), SW_THREADS, SW_SMEM, s>>>(p, my, mp);
    LCHECK();
    const size_t smem = (size_t)OV_ROWS * K * 4;
    e = cudaFuncSetAttribute(screen_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    screen_rows_kernel<<<(unsigned)(2 * sms), 256, smem, s>>>(X, n, D, K, margin, (long long)(max_marks * (double)n), mu, w2, c2d, b.ovf,
                                                              b.pt_off, b.pt_cnt, b.ids, b.ctl);
    *launches += 3;
    return cudaGetLastError();
}

cudaError_t launch_screen_eval(cudaStream_t s, int mode, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                               const double* c2d, const ScreenBuffers& b, float* logp, int32_t* idx) {
    const unsigned blocks = (unsigned)((n + SCR_RANGE - 1) / SCR_RANGE);
    const size_t smem = (size_t)K * 4;
    if (mode == SCREEN_EM)
        screen_eval_kernel<SCREEN_EM><<<blocks, 256, smem, s>>>(X, n, D, K, mu, w2, c2d, b.pt_off, b.pt_cnt, b.ids, b.val, b.counts, b.ll, nullptr, nullptr, b.ctl);
    else if (mode == SCREEN_LOGP)
        screen_eval_kernel<SCREEN_LOGP><<<blocks, 256, 0, s>>>(X, n, D, K, mu, w2, c2d, b.pt_off, b.pt_cnt, b.ids, b.val, nullptr, b.ll, logp, nullptr, b.ctl);
    else
        screen_eval_kernel<SCREEN_ARGMAX><<<blocks, 256, smem, s>>>(X, n, D, K, mu, w2, c2d, b.pt_off, b.pt_cnt, b.ids, b.val, b.counts, nullptr, nullptr, idx, b.ctl);
    return cudaGetLastError();
}

cudaError_t launch_screen_stats(cudaStream_t s, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                                const double* c2d, const ScreenBuffers& b, double* Nk, double* S1, double* S2, int64_t* launches) {
    const int blocks = (int)((n + SCR_RANGE - 1) / SCR_RANGE);
    screen_scan_kernel<<<(K + 31) / 32, 1024, 0, s>>>(b.counts, blocks, K, b.totals, b.off, b.segoff, b.ctl);
    LCHECK();
    const int K2 = (K + 1) & ~1;
    const size_t smem = (size_t)K2 * 4 + (size_t)K2 * 16;
    cudaError_t e = cudaFuncSetAttribute(screen_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    screen_fill_kernel<<<blocks, 256, smem, s>>>(n, K, b.pt_off, b.pt_cnt, b.ids, b.val, b.counts, b.off, b.srt, b.ctl);
    LCHECK();
    int lpr = 1;
    while (4 * lpr < D) lpr <<= 1;
    screen_stats_kernel<<<148 * 6, 256, (size_t)(K + 1) * 4, s>>>(X, D, lpr, mu, w2, b.srt, b.off, b.segoff, K, b.part, b.ctl);
    LCHECK();
    screen_reduce_kernel<<<K, 1024, 0, s>>>(D, K, b.part, b.segoff, mu, c2d, Nk, S1, S2, b.ll + SCR_LL, b.ctl);
    *launches += 4;
    return cudaGetLastError();
}

}  // namespace fg
