// esb_qat.cu -- kernels of the quantisation-aware training step of
// Algorithm 1 (DNN training with ESB):
//   * DN followed by ESB projection (Sec. III-D "Normalization": x_hat =
//     (x - mu) / (sigma + eps), eps = 1e-7; the normalised data meet the
//     DDA scale alpha*(b,k) directly), emitting the codes and the
//     fake-quantised values alpha* q the forward pass multiplies;
//   * the backward pass through it: the straight-through estimator (the
//     gradient w.r.t. the normalised data passes the projection unchanged,
//     Algorithm 1 multiplies no derivative of ESB) and the exact derivative
//     of DN, whose mean and sigma depend on every element:
//       dL/dx_j = (g_j - mean(g)) / s - c_j sum_i(g_i c_i) / (d sigma s^2),
//     c = x - mu, s = sigma + eps;
//   * the exponential moving average of the activation statistics
//     (Sec. III-D: mu <- (1 - gamma) mu + gamma mu_i, likewise sigma).
// GB300 runs fp64 at a small fraction of its fp32 rate, so the element-wise
// work and each thread's sums use unevaluated pairs of fp32 numbers (~48
// significant bits, error-free transformations); fp64 joins the threads'
// sums and computes the scalars.  Values that pairs cannot carry (not
// finite, or so small that a product's error term would underflow) are
// recomputed in fp64.  The order of every sum is fixed, so results are
// reproducible.
#include <cstdint>
#include <cuda_runtime.h>

#include "esb_common.cuh"
#include "esb_internal.h"

namespace esb {

namespace {

constexpr int kQatThreads = 256;

// x_hat = fl32(fl32(x - mu) / fl32(sigma + eps)), then its projection with
// scale alpha*; codes packed cpw per word (rows of ldc words, cols codes).
//
// fl32(c / s) is monotone in c, so the projection's thresholds T_j on x_hat
// become thresholds on |c| = |fl32(x - mu)|: the smallest float whose
// quotient by s reaches T_j, found once per block with the same division.
// No division per element (but for few elements of a wide format, see
// launch_dn_project), and the fake-quantised value is a table entry.
// HBM-bound (4 B in, 4.5 B out per element at b = 4): a warp loads and
// stores 128 consecutive values at a time.  6.4 M elements, (4,2): 31.8 us with
// one thread per word and a division per element, 12.7 us this way (inputs in
// L2; 34 and 18 us from HBM).
template <int B>
struct DnTable {
    static constexpr int CAP = B <= 6 ? 1024 : 2048;
    float T[128];
    uint2 cells[B == 4 ? 1 : CAP];
    float xq[1 << B];
};

constexpr int kDnUnroll = 6;       // granules in flight per warp (flat 4-bit path)

template <int B>
__global__ void __launch_bounds__(kQatThreads)
dn_project_kernel(const float* __restrict__ x, int64_t rows, int64_t cols, const double* __restrict__ stats,
                  float alpha, ProjParams p, uint32_t* __restrict__ codes, int64_t ldc, float* __restrict__ xq, int flat, int divide)
{
    constexpr int CPW = 32 / B;
    constexpr int L = 1 << (B - 1);
    __shared__ DnTable<B> sm;
    griddep_wait();                                   // x and stats may come from the previous launch
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // fp64 in one thread: its pipe would serve every warp of the SM in turn
    __shared__ float2 ms;
    if (threadIdx.x == 0) ms = make_float2((float)__ldg(stats), (float)(__ldg(stats + 1) + 1e-7));
    if (threadIdx.x < (1 << B)) sm.xq[threadIdx.x] = __fmul_rn(alpha, code_value(threadIdx.x, B, p.k));
    build_thresholds(sm.T, p, alpha, warp, lane, 0, kQatThreads / 32);
    __syncthreads();
    const float m = ms.x, s = ms.y;
    // also for a sigma that is not finite (or +-0 with eps lost), which no threshold can stand for
    const bool by_div = divide || !(s > 0.0f && s < __int_as_float(0x7f800000));
    if (!by_div) {
        for (int j = warp; j < L - 1; j += kQatThreads / 32) {
            const float t = sm.T[j];                  // each threshold is read and replaced by one warp
            const float tc = t < __int_as_float(0x7f800000) ? warp_threshold(s, t, false, lane) : t;
            __syncwarp();
            if (lane == 0) sm.T[j] = tc;
        }
    }
    __syncthreads();
    Thr7 t7;
#pragma unroll
    for (int i = 0; i < 7; i++) t7.t[i] = B == 4 ? sm.T[i] : 0.0f;
    int h0 = 0, hmax = 0;
    const bool by_cells = B != 4 && !by_div && build_cells<B, DnTable<B>::CAP>(sm.cells, h0, hmax, sm.T, p);
    const int sh = cell_shift(p.k);
    const uint32_t amask = p.is_signed ? 0x7fffffffu : 0xffffffffu;
    auto code_of = [&](float v) -> uint32_t {
        const float c = __fsub_rn(v, m);
        if (by_div) return project_by_table_t<B>(__fdiv_rn(c, s), sm.T, p);
        if (B == 4) return project_by_thr7(c, t7, p);
        return by_cells ? project_by_cells<B>(c, sm.cells, h0, hmax, sh, amask) : project_by_table_t<B>(c, sm.T, p);
    };
    const int64_t gwarp = (int64_t)blockIdx.x * (kQatThreads / 32) + warp;
    const int64_t nwarps = (int64_t)gridDim.x * (kQatThreads / 32);
    if (B == 4 && flat) {
        // granules of 128 values: lane l takes values 4l .. 4l + 3, lane
        // pairs join their halves of a code word
        const int64_t n = rows * cols;                // a multiple of 8
        const int64_t gran = (n + 127) / 128;
        for (int64_t g0 = gwarp; g0 < gran; g0 += kDnUnroll * nwarps) {
            float4 v[kDnUnroll];
#pragma unroll
            for (int u = 0; u < kDnUnroll; u++) {
                const int64_t e = (g0 + u * nwarps) * 128 + 4 * lane;
                v[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (e < n) v[u] = __ldg(reinterpret_cast<const float4*>(x + e));
            }
#pragma unroll
            for (int u = 0; u < kDnUnroll; u++) {
                const int64_t e = (g0 + u * nwarps) * 128 + 4 * lane;
                const bool in = e < n;
                const float q[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                uint32_t h = 0u;
                if (by_div) {
#pragma unroll
                    for (int i = 0; i < 4; i++) h |= code_of(q[i]) << (4 * i);
                } else {
                    uint32_t J = 0u, S = 0u;
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const float c = __fsub_rn(q[i], m);
                        J |= bucket7(p.is_signed ? fabsf(c) : c, t7) << (4 * i);
                        S |= ((__float_as_uint(c) >> 31) & (uint32_t)p.is_signed) << (4 * i + 3);
                    }
                    h = codes8_b4(J, S, p.k) & 0xffffu;
                }
                if (xq && in)
                    *reinterpret_cast<float4*>(xq + e) = make_float4(sm.xq[h & 15u], sm.xq[(h >> 4) & 15u],
                                                                     sm.xq[(h >> 8) & 15u], sm.xq[h >> 12]);
                const uint32_t other = __shfl_down_sync(0xffffffffu, h, 1);
                if (in && (lane & 1) == 0) codes[e >> 3] = h | (other << 16);
            }
        }
        return;
    }
    // general path: a thread per word (warp segments packed through shared
    // memory took 176 us against 95 for a training step of rows of 17 values)
    {
        const int64_t total = rows * ldc, stride = (int64_t)gridDim.x * blockDim.x;
        for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total; u += stride) {
            const int64_t r = u < (1ll << 32) && ldc < (1ll << 31) ? (int64_t)((uint32_t)u / (uint32_t)ldc) : u / ldc;
            const int64_t c0 = (u - r * ldc) * CPW;
            const float* xr = x + r * cols + c0;
            uint32_t word = 0u;
#pragma unroll
            for (int j = 0; j < CPW; j++) {
                uint32_t code = p.zero_code;
                if (c0 + j < cols) {
                    code = code_of(__ldg(xr + j));
                    if (xq) xq[r * cols + c0 + j] = sm.xq[code];
                }
                word |= code << (B * j);
            }
            codes[u] = word;
        }
    }
}

// ------------------------------------------------------------- backward
//
// fp32 pairs: the scalars as (hi, lo) from their fp64 values.
struct F2 { float h, l; };
__device__ __forceinline__ F2 f2_of(double d)
{
    F2 r;
    r.h = (float)d;
    r.l = (float)(d - (double)r.h);
    return r;
}
// v - a, exact in the high part's rounding error
__device__ __forceinline__ F2 f2_sub(float v, const F2& a)
{
    const float d = v - a.h;
    const float bp = d - v;
    F2 r;
    r.h = d;
    r.l = ((v - (d - bp)) - (a.h + bp)) - a.l;
    return r;
}
__device__ __forceinline__ F2 f2_mul(const F2& a, const F2& b)
{
    F2 r;
    r.h = __fmul_rn(a.h, b.h);                        // never contracted into a later add: its error term follows
    r.l = fmaf(a.h, b.h, -r.h) + fmaf(a.h, b.l, a.l * b.h);
    return r;
}
// Scalars that a pair holds to 2^-48 and whose products with ordinary values
// stay well inside fp32's range.
__device__ __forceinline__ bool f2_safe(double d) { return d == 0.0 || (fabs(d) > 0x1p-100 && fabs(d) < 0x1p60); }

constexpr int kGradUnroll = 4;

// Per-block partials of sum g and sum g (x - mu), in a fixed order: a
// thread's elements (float4 when both pointers are 16-byte aligned) in fp32
// pairs, the block's warps in fp64.  Reads 8 B per element; with fp64 per
// element it took 67 us for 6.4 M elements from HBM, bound by the fp64 pipe;
// 16 us now.
__global__ void __launch_bounds__(kQatThreads)
dn_grad_partials_kernel(const float* __restrict__ g, const float* __restrict__ x, int64_t n,
                        const double* __restrict__ stats, double2* __restrict__ part, int vec)
{
    __shared__ double2 sh[kQatThreads / 32];
    __shared__ F2 sh_mu;
    __shared__ float sh_gmin;
    griddep_wait();
    if (threadIdx.x == 0) {                           // fp64 in one thread (see dn_project_kernel)
        const double mu = __ldg(stats), sigma = __ldg(stats + 1);
        sh_mu = f2_of(mu);
        // a thread's largest |g| for which the error terms of its products
        // g (x - mu), about 2^-24 |g| sigma, stay above the subnormals
        const bool ok = sigma > 0x1p-40 && sigma < 0x1p40 && fabs(mu) < 0x1p60;
        sh_gmin = ok ? (float)fmax(0x1p-100, 0x1p-100 / sigma) : __int_as_float(0x7f800000);
    }
    __syncthreads();
    const F2 mu2 = sh_mu;
    const float gmin = sh_gmin;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float s1h = 0.0f, s1l = 0.0f, s2h = 0.0f, s2l = 0.0f, mx = 0.0f;
    auto add = [&](float gi, float xi) {
        mx = fmaxf(mx, fabsf(gi));
        df_add(s1h, s1l, gi);
        const F2 c = f2_sub(xi, mu2);
        const float ph = __fmul_rn(gi, c.h);
        s2l += fmaf(gi, c.h, -ph) + gi * c.l;
        df_add(s2h, s2l, ph);
    };
    const int64_t nv = vec ? n / 4 : 0;
    const float4* g4 = reinterpret_cast<const float4*>(g);
    const float4* x4 = reinterpret_cast<const float4*>(x);
    for (int64_t i0 = t0; i0 < nv; i0 += kGradUnroll * stride) {
        float4 a[kGradUnroll], b[kGradUnroll];
#pragma unroll
        for (int u = 0; u < kGradUnroll; u++) {
            const int64_t i = i0 + u * stride;
            a[u] = b[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i < nv) { a[u] = __ldg(g4 + i); b[u] = __ldg(x4 + i); }
        }
#pragma unroll
        for (int u = 0; u < kGradUnroll; u++) {
            if (i0 + u * stride >= nv) break;
            add(a[u].x, b[u].x); add(a[u].y, b[u].y); add(a[u].z, b[u].z); add(a[u].w, b[u].w);
        }
    }
    for (int64_t i = nv * 4 + t0; i < n; i += stride) add(g[i], x[i]);
    auto finite = [&]() { return fabsf(s1h + s1l) < __int_as_float(0x7f800000) && fabsf(s2h + s2l) < __int_as_float(0x7f800000); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    bool pairs = __all_sync(0xffffffffu, finite() && gmin < 1.0f && (mx == 0.0f || mx > gmin));
    if (pairs) {
        // the warp's sums in pairs; fp64 only once per warp (its pipe takes
        // a block's worth of conversions and adds longer than the loads).
        // Lanes whose own sums are finite can still overflow together.
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float a = __shfl_xor_sync(0xffffffffu, s1h, o), b = __shfl_xor_sync(0xffffffffu, s1l, o);
            const float c = __shfl_xor_sync(0xffffffffu, s2h, o), d = __shfl_xor_sync(0xffffffffu, s2l, o);
            df_add(s1h, s1l, a); s1l += b;
            df_add(s2h, s2l, c); s2l += d;
        }
        pairs = __all_sync(0xffffffffu, finite());
    }
    if (pairs) {
        if (lane == 0) sh[warp] = make_double2((double)s1h + (double)s1l, (double)s2h + (double)s2l);
    } else {                                          // this warp's elements again in fp64
        const double mu = __ldg(stats);
        double s1 = 0.0, s2 = 0.0;
        auto add64 = [&](int64_t i) {
            const double gi = (double)g[i];
            s1 += gi;
            s2 = fma(gi, (double)x[i] - mu, s2);
        };
        for (int64_t i = t0; i < nv; i += stride)
            for (int j = 0; j < 4; j++) add64(4 * i + j);
        for (int64_t i = nv * 4 + t0; i < n; i += stride) add64(i);
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) sh[warp] = make_double2(s1, s2);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 t = sh[0];
        for (int w = 1; w < kQatThreads / 32; w++) { t.x += sh[w].x; t.y += sh[w].y; }
        part[blockIdx.x] = t;
    }
}

// The scalars of dn_grad_kernel, by one block: the partials in index order,
// then the quotients.  One block, because fp64 divisions in every block of
// the element-wise kernel cost it 20 us.
struct GradScalars {
    double mu, s, gm, k2;                             // for the elements fp64 recomputes
    F2 mu2, gm2, k22, inv2;
    int safe, none;                                   // none: mean and k2 are zero (no gradient at all)
};
__global__ void __launch_bounds__(kQatThreads)
dn_grad_total_kernel(double2* part, int nparts, int64_t n, const double* __restrict__ stats)
{
    __shared__ double2 sh[kQatThreads / 32];
    griddep_wait();
    double s1 = 0.0, s2 = 0.0;
    for (int i = threadIdx.x; i < nparts; i += kQatThreads) { s1 += part[i].x; s2 += part[i].y; }
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = make_double2(s1, s2);
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 t = sh[0];
        for (int w = 1; w < kQatThreads / 32; w++) { t.x += sh[w].x; t.y += sh[w].y; }
        const double sigma = __ldg(stats + 1), s = sigma + 1e-7, d = (double)n;
        part[nparts] = make_double2(t.x / d, sigma > 0.0 ? t.y / (d * sigma * s * s) : 0.0);
    }
}

// dL/dx of every element.  HBM-bound: 8 B in, 4 B out per element.  6.4 M
// elements from HBM: 174 us with an fp64 division per element, 18 us now.
__global__ void __launch_bounds__(kQatThreads)
dn_grad_kernel(const float* __restrict__ g, const float* __restrict__ x, int64_t n, const double* __restrict__ stats,
               const double2* __restrict__ tot, float* __restrict__ gx, int vec)
{
    __shared__ GradScalars sc;
    griddep_wait();
    if (threadIdx.x == 0) {
        const double2 t = __ldcg(tot);
        const double mu = __ldg(stats), s = __ldg(stats + 1) + 1e-7;
        const double inv = 1.0 / s;
        sc.mu = mu; sc.s = s; sc.gm = t.x; sc.k2 = t.y;
        sc.mu2 = f2_of(mu); sc.gm2 = f2_of(t.x); sc.k22 = f2_of(t.y); sc.inv2 = f2_of(inv);
        sc.safe = f2_safe(mu) && f2_safe(t.x) && f2_safe(t.y) && f2_safe(inv) && inv != 0.0;
        sc.none = sc.safe && t.x == 0.0 && t.y == 0.0;
    }
    __syncthreads();
    const bool safe = sc.safe != 0;
    const F2 mu2 = sc.mu2, gm2 = sc.gm2, k22 = sc.k22, inv2 = sc.inv2;
    auto one = [&](float gi, float xi) -> float {
        const F2 a = f2_mul(f2_sub(gi, gm2), inv2);
        const F2 b = f2_mul(f2_sub(xi, mu2), k22);
        const F2 r = f2_sub(a.h, b);                  // a.h - (b.h + b.l)
        const float y = r.h + (r.l + a.l);
        // not finite, or small enough that an error term may have underflowed
        if (!safe || !(fabsf(y) > 0x1p-100f) || !(fabsf(y) < __int_as_float(0x7f800000))) {
            if (sc.none && __float_as_uint(gi) == 0u && fabsf(xi) < __int_as_float(0x7f800000)) return 0.0f;
            return (float)(((double)gi - sc.gm) / sc.s - ((double)xi - sc.mu) * sc.k2);
        }
        return y;
    };
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nv = vec ? n / 4 : 0;
    constexpr int U = 3;
    for (int64_t i0 = t0; i0 < nv; i0 += U * stride) {
        float4 a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            a[u] = b[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i0 + u * stride < nv) {
                a[u] = __ldg(reinterpret_cast<const float4*>(g) + i0 + u * stride);
                b[u] = __ldg(reinterpret_cast<const float4*>(x) + i0 + u * stride);
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i0 + u * stride < nv)
                reinterpret_cast<float4*>(gx)[i0 + u * stride] =
                    make_float4(one(a[u].x, b[u].x), one(a[u].y, b[u].y), one(a[u].z, b[u].z), one(a[u].w, b[u].w));
    }
    for (int64_t i = nv * 4 + t0; i < n; i += stride) gx[i] = one(g[i], x[i]);
}

// mu <- (1 - gamma) mu + gamma mu_i; sigma likewise (products and sums
// rounded separately, no fused multiply-add).
__global__ void ema_kernel(const double* __restrict__ batch, double* __restrict__ running, double gamma)
{
    if (threadIdx.x < 2) {
        const double a = __dmul_rn(1.0 - gamma, running[threadIdx.x]);
        const double b = __dmul_rn(gamma, batch[threadIdx.x]);
        running[threadIdx.x] = __dadd_rn(a, b);
    }
}

int qat_blocks(int64_t units)
{
    int64_t b = (units + kQatThreads - 1) / kQatThreads;
    const int64_t cap = (int64_t)device_sm_count() * 4;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

size_t dn_grad_workspace_bytes(int64_t n) { return sizeof(double2) * (size_t)(qat_blocks(n) + 1); }

cudaError_t launch_dn_project(const float* x, int64_t rows, int64_t cols, const double* stats, int b, int k,
                              int is_signed, int rounding, float alpha, uint32_t* codes, int64_t ldc, float* xq,
                              cudaStream_t st)
{
    const ProjParams p = make_proj_params(b, k, is_signed, rounding);
    auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    const int flat = b == 4 && ldc * 8 == cols && al16(x) && (!xq || al16(xq));
    const int64_t sms = device_sm_count(), words = rows * ldc;
    // Every block builds its tables, and all of an SM's blocks at once take
    // longer over it than a block alone: no more blocks than have work.  Flat
    // 4-bit codes: a warp's granules in flight together (20000 x 64: 4.7 us,
    // 12.4 with a granule per warp).  Elsewhere a cap by width (20000 x 64, 8
    // bits: 12.8 us with 2 blocks an SM, 16.5 with 4, 26.2 with 8; 100352 x 64, 6
    // bits: 27.8, 24.6, 24.5; 2 bits: 33.4, 37.4, 42.6; 100352 x 77, 4 bits: 39.6,
    // 43.9, 37.2).
    const int64_t cap = sms * (b == 2 || b == 8 ? 2 : (b == 4 ? 8 : 4));
    int64_t blocks = flat ? (rows * cols / 128 + 8 * kDnUnroll - 1) / (8 * kDnUnroll) : (words + kQatThreads - 1) / kQatThreads;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    // Wide formats with few words per thread: a division per element costs less
    // than thresholds on |x - mu| and their table (1000 x 77, 8 bits: 6.0 us against
    // 8.3 to 9.6; 6 bits 3.9 against 4.3 to 4.7; 10000 x 64, 8 bits 9.7 against 10.8
    // to 12.3; at 20000 x 64, 320000 words, they are level; at 100352 x 64 the table
    // takes 24.6 against 27.8 at 6 bits).
    const int divide = b >= 6 && words <= sms * 8 * kQatThreads;
    using Kernel = void (*)(const float*, int64_t, int64_t, const double*, float, ProjParams, uint32_t*, int64_t, float*, int, int);
    static const Kernel kernels[] = {dn_project_kernel<2>, dn_project_kernel<3>, dn_project_kernel<4>, dn_project_kernel<5>,
                                     dn_project_kernel<6>, dn_project_kernel<7>, dn_project_kernel<8>};
    return launch_pdl(kernels[b - 2], dim3((unsigned)blocks), dim3(kQatThreads), 0, st, x, rows, cols, stats, alpha, p,
                      codes, ldc, xq, flat, divide);
}

cudaError_t launch_dn_grad(const float* g, const float* x, int64_t n, const double* stats, void* workspace, float* gx,
                           cudaStream_t st)
{
    const int nb = qat_blocks(n);
    double2* part = static_cast<double2*>(workspace);
    auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    const int vec = al16(g) && al16(x);
    cudaError_t e = launch_pdl(dn_grad_partials_kernel, dim3((unsigned)nb), dim3(kQatThreads), 0, st, g, x, n, stats, part, vec);
    if (e != cudaSuccess) return e;
    e = launch_pdl(dn_grad_total_kernel, dim3(1), dim3(kQatThreads), 0, st, part, nb, n, stats);
    if (e != cudaSuccess) return e;
    return launch_pdl(dn_grad_kernel, dim3((unsigned)qat_blocks(vec ? n / 4 : n) * 2), dim3(kQatThreads), 0, st, g, x, n,
                      stats, (const double2*)(part + nb), gx, vec && al16(gx) ? 1 : 0);
}

cudaError_t launch_ema(const double* batch, double* running, double gamma, cudaStream_t st)
{
    ema_kernel<<<1, 32, 0, st>>>(batch, running, gamma);
    return cudaGetLastError();
}

}  // namespace esb
