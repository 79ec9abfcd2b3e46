// esb_conv_stem.cu -- strided ESB convolution of images with up to 4
// channels (the first layer of a network: 7x7/2, 3x3/2, 11x11/4; Sec. IV-B).
//
// A pixel's codes decode to 4 E4M3 bytes, so the taps of one filter row are
// 4 S contiguous bytes of a decoded input row, and im2col is only a matter of
// where a row of the MMA operand starts: output q reads from byte 4 (stride q
// - pad).  That is 16-byte aligned, as the K-major no-swizzle layout needs,
// for every q = phi i + f of one residue f modulo phi = 4 / stride.  So each
// input row is decoded once into phi copies, copy f shifted by stride f
// pixels, U 16-byte units apart; tile row f U + i is output phi i + f of one
// output row, its K chunk g (4 taps) unit f U + i + g, and the whole operand of
// filter row r is that decoded row seen through a descriptor with SBO = 128
// and LBO = 16 bytes (the chunks overlap).  K = R rows x G chunks, G even; the
// filter's bytes past S taps or past the channels are zero.  Tile rows with i
// past the segment's outputs compute on neighbouring units and are not stored.
//
// A CTA walks consecutive output rows, and decoded rows live in a ring of NR
// slots: the next output row of the same image needs only `stride` new input
// rows.  Each row has its own full and empty barrier; the MMA warp's commits
// free the rows that the next tile does not use.
//
// 224 x 224 x 3, 7x7/2 -> 64, batch 64, 4-bit: 372 us on the im2col kernel
// (49 single words gathered and decoded per output pixel, 5 of the 8 K slots
// of each word padding), 86 us here; 3x3/2 -> 32: 53 us (69 while the decoders
// stepped through every row and divided for every tile).
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "esb_tc.cuh"

namespace esb {

namespace {

constexpr int kStemMaxRing = 24;

struct StemGeom {
    const uint32_t* X;
    int ldx, H, W, P, Q, R, S, C, stride, pad;
    int phi;             // output residues per 16-byte step: 4 / stride
    int G;               // 16-byte chunks (4 taps) per filter row, even
    int Ui;              // outputs of one residue per segment
    int U;               // units of one copy: Ui + G - 1
    int nseg;            // column segments per output row
    int pitch;           // bytes of a ring slot: 128 + G - 1 units
    int NR;              // ring slots
};

// Input pixel word -> its (up to 4) codes as E4M3 bytes, channel order.
template <int B>
__device__ __forceinline__ uint32_t stem_pixel(uint32_t w, int k)
{
    return e4m3_4<B>(spread4<B>(rot_word<B>(w, k)), k);
}

// One input row by one warp: lane l takes pixel positions l, l + 32, ... of a
// batch of 32 * kStemUn.  Loaded ahead of its slot, then each pixel is decoded
// and stored to its place in every copy (position j is pixel j - stride f of
// copy f).
constexpr int kStemUn = 8;

struct StemRow {                     // row h (of image n), pixel x0 at position 0
    const uint32_t* x;               // first pixel of the row; nullptr: outside the image
    int x0;
};

__device__ __forceinline__ void stem_load(const StemGeom& g, const StemRow& row, int j0, int lane, uint32_t zw,
                                          uint32_t (&w)[kStemUn])
{
#pragma unroll
    for (int u = 0; u < kStemUn; u++) {
        const int x = row.x0 + j0 + 32 * u + lane;
        w[u] = zw;
        if (row.x && (unsigned)x < (unsigned)g.W) w[u] = __ldg(row.x + (int64_t)x * g.ldx);
    }
}

template <int B>
__device__ __forceinline__ void stem_store(const StemGeom& g, int j0, uint8_t* slot, int lane, int k, uint32_t cmask,
                                           const uint32_t (&w)[kStemUn])
{
    const int n4 = 4 * g.U;                           // positions of a copy
    uint8_t* const p0 = slot + (j0 + lane) * 4;
    const int f1 = g.U * 16 - 4 * g.stride;           // from copy 0 to copy 1
#pragma unroll
    for (int u = 0; u < kStemUn; u++) {
        const int j = j0 + 32 * u + lane;
        const uint32_t v = stem_pixel<B>(w[u], k) & cmask;
        if (j < n4) *reinterpret_cast<uint32_t*>(p0 + 128 * u) = v;
        if (g.phi > 1 && (unsigned)(j - g.stride) < (unsigned)n4) *reinterpret_cast<uint32_t*>(p0 + 128 * u + f1) = v;
    }
}

// Filter chunk c (row r = c / G, taps 4 (c % G) ..) of output channel row n.
template <int B>
__device__ __forceinline__ void stem_filter(const StemGeom& g, const uint32_t* W, int64_t ldw, int64_t n, int64_t N, int c, int k,
                                            uint32_t cmask, uint8_t* sB, int BN, int row)
{
    uint32_t o[4] = {0u, 0u, 0u, 0u};
    const int r = c / g.G, s0 = (c - r * g.G) * 4;
    if (n < N && r < g.R) {
        const uint32_t* p = W + ((n * g.R + r) * g.S + s0) * ldw;
#pragma unroll
        for (int t = 0; t < 4; t++)
            if (s0 + t < g.S) o[t] = stem_pixel<B>(__ldg(p + t * ldw), k) & cmask;
    }
    *reinterpret_cast<uint4*>(sB + (c >> 3) * BN * kBK + swz(row, c & 7)) = make_uint4(o[0], o[1], o[2], o[3]);
}

}  // namespace

template <int EPI>
__global__ void __launch_bounds__(kWsThreads, 1)
esb_conv_stem_kernel(StemGeom g, const uint32_t* Wt, int64_t ldw, int64_t N, OpFmt fa, OpFmt fb, int BN, int nkb, int n_tiles,
                     int m_tiles, float acc_scale, const __grid_constant__ EpiParams ep)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sB = smem;                                        // nkb blocks of BN x 128 bytes (SW128)
    uint8_t* sA = sB + nkb * BN * kBK;                         // NR decoded rows
    float* thr = reinterpret_cast<float*>(sA + g.NR * g.pitch);
    uint64_t* full = reinterpret_cast<uint64_t*>(thr + 128);
    uint64_t* empty = full + kStemMaxRing;
    uint64_t* tfull = empty + kStemMaxRing;
    uint64_t* tempty = tfull + kMaxAcc;
    uint64_t* drain = tempty + kMaxAcc;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* err = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x;
    const int warp = warp_index(), lane = tid & 31;
    const int n_tile = (int)(blockIdx.x % n_tiles);
    const int cta = blockIdx.x / n_tiles, ctas = gridDim.x / n_tiles;
    const int64_t n0 = (int64_t)n_tile * BN;
    // consecutive tiles: (image, segment, output row), the row fastest
    const int t_lo = (int)((int64_t)m_tiles * cta / ctas), t_hi = (int)((int64_t)m_tiles * (cta + 1) / ctas);
    const int lacc = acc_buffers_log2(BN);
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < (BN << lacc)) tmem_cols <<= 1;
    const EpiSplit sp = epi_split<EPI>(ep, BN, t_hi - t_lo);
    // the layout above must fit the dynamic allocation (uniform for the CTA)
    if ((uintptr_t)(reinterpret_cast<const volatile uint8_t*>(err) + 4 - smem_raw) > dynamic_smem_bytes()) {
        if (tid == 0) record_status(ep.status, ESB_ERR_INTERNAL);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < g.NR; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < (1 << lacc); a++) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], sp.tempty_count());
        }
        mbar_init(drain, 1);
        *err = 0;
        fence_mbar_init();
    }
    ws_alloc(warp, tmem_slot, tmem_cols);
    __syncthreads();                                  // barriers initialised, TMEM allocated
    griddep_wait();                                   // X, W and the alphas may come from the previous launch

    // padding slots of a pixel's word must not count even if they are not zero codes
    const uint32_t cmask = g.C >= 4 ? 0xffffffffu : (1u << (8 * g.C)) - 1u;
    const int nnew = g.stride < g.R ? g.stride : g.R; // rows a following output row adds
    constexpr int kSetup = kWsProdWarp0 * 32;
    if (warp < kWsProdWarp0) {
        // filters: one 16-byte chunk per thread and pass
        with_width(fb.b, [&](auto width) {
            for (int i = tid; i < nkb * 8 * BN; i += kSetup) {
                const int row = i >> 3, c = i & 7;
                const int kb = row / BN;
                stem_filter<decltype(width)::value>(g, Wt, ldw, n0 + (row - kb * BN), N, kb * 8 + c, fb.k, cmask, sB, BN,
                                                    row - kb * BN);
            }
        });
        fence_proxy_async_smem();
        if (warp == kWsMmaWarp) {
            asm volatile("bar.sync 1, %0;" ::"n"(kSetup) : "memory");
        } else {
            asm volatile("bar.arrive 1, %0;" ::"n"(kSetup) : "memory");
            ws_thresholds(thr, ep, warp, lane);
        }
    }
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp >= kWsProdWarp0) {
        // ---------------------------------------------- row decoders: row rho by warp rho % 7
        const int pw = warp - kWsProdWarp0;
        with_width(fa.b, [&](auto width) {
            constexpr int B = decltype(width)::value;
            const uint32_t zw = fmt_zero_word(B, fa.k);
            const int npos = 4 * g.U + g.stride * (g.phi - 1);
            // cursor of this warp's next row: tile T (output row p of strip
            // `strip`), filter row r, ring slot s and its phase
            int T = t_lo, strip = t_lo / g.P, p = t_lo - strip * g.P, r = 0, s = 0;
            uint32_t ph = 0u;
            auto skip = [&](int rows) {               // `rows` rows on in the sequence
                s += rows;
                if (s >= g.NR) { s -= g.NR; ph ^= 1u; }
                while (rows > 0) {
                    const int left = g.R - r;
                    if (rows < left) { r += rows; break; }
                    rows -= left;
                    T++;
                    r = g.R - nnew;
                    if (++p == g.P) { p = 0; strip++; r = 0; }
                }
            };
            auto row_at = [&]() -> StemRow {
                const int n = g.nseg == 1 ? strip : strip / g.nseg, seg = g.nseg == 1 ? 0 : strip - n * g.nseg;
                const int h = p * g.stride - g.pad + r;
                StemRow q;
                q.x = (unsigned)h < (unsigned)g.H ? g.X + ((int64_t)n * g.H + h) * g.W * g.ldx : nullptr;
                q.x0 = g.stride * g.phi * seg * g.Ui - g.pad;
                return q;
            };
            skip(pw);
            uint32_t w[kStemUn];
            StemRow row;
            if (T < t_hi) { row = row_at(); stem_load(g, row, 0, lane, zw, w); }
            while (T < t_hi) {
                if (!wait_or_abort(&empty[s], ph ^ 1u, err)) { *err = 1; break; }
                uint8_t* const slot = sA + s * g.pitch;
                uint64_t* const done = &full[s];
                // the batches of this row, then the next row's first one
#pragma unroll 1
                for (int j0 = 0; j0 < npos; j0 += 32 * kStemUn) {
                    uint32_t wn[kStemUn];
                    const bool more = j0 + 32 * kStemUn < npos;
                    if (!more) {
                        skip(kWsProdWarps);
                        if (T < t_hi) row = row_at(); else row.x = nullptr;
                    }
                    stem_load(g, row, more ? j0 + 32 * kStemUn : 0, lane, zw, wn);
                    stem_store<B>(g, j0, slot, lane, fa.k, cmask, w);
#pragma unroll
                    for (int u = 0; u < kStemUn; u++) w[u] = wn[u];
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(done);
            }
        });
    } else if (warp == kWsMmaWarp) {
        // ---------------------------------------------- MMA issue
        const uint32_t idesc = idesc_e4m3_f32(BN);
        const uint32_t leader = elect_one();
        const uint64_t a_desc = smem_desc_noswz(smem_u32(sA), 16u, 128u), b_desc = smem_desc_sw128(smem_u32(sB));
        const uint32_t a_step = (uint32_t)g.pitch >> 4, b_step = (uint32_t)(BN * kBK) >> 4;
        const int steps = g.G >> 1;
        int s = 0, base = 0;                          // next row to arrive; the tile's first row (ring slots)
        uint32_t ph = 0u;
        int p = t_lo % g.P;
        bool ok = true;
        for (int T = t_lo; T < t_hi && ok; T++) {
            const int i = T - t_lo, a = i & ((1 << lacc) - 1);
            ok = warp_wait(&tempty[a], (uint32_t)((i >> lacc) & 1) ^ 1u, err);
            if (!ok) break;
            const int add = (i == 0 || p == 0) ? g.R : nnew;
            if (add == g.R) base = s;
            for (int j = 0; j < add && ok; j++) {
                ok = warp_wait(&full[s], ph, err);
                if (++s == g.NR) { s = 0; ph ^= 1u; }
            }
            if (!ok) break;
            tc_fence_after();
            const uint32_t d = tmem_base + (uint32_t)(a * BN);
            uint32_t acc = 0u, kq = 0u;
            int slot = base;
            for (int r = 0; r < g.R; r++) {
                const uint64_t ad = a_desc + (uint64_t)((uint32_t)slot * a_step);
                for (int j = 0; j < steps; j++, kq++) {
                    mma_f8f6f4(d, ad + (uint64_t)(2 * j), b_desc + (uint64_t)((kq >> 2) * b_step + (kq & 3u) * 2u), idesc, acc,
                               leader);
                    acc = 1u;
                }
                if (++slot == g.NR) slot = 0;
            }
            mma_commit(&tfull[a], leader);
            // rows the next tile does not use (all of them at the end of an image's segment)
            if (++p == g.P) p = 0;
            const int rel = (T + 1 == t_hi || p == 0) ? g.R : nnew;
            for (int j = 0; j < rel; j++) {
                mma_commit(&empty[base], leader);
                if (++base == g.NR) base = 0;
            }
        }
        if (!ok) *err = 1;
        ws_drain(drain, err, leader);
    } else if (warp < sp.warps) {
        // ---------------------------------------------- epilogue
        const int row = (warp & 3) * 32 + lane;
        const int f = row / g.U, i = row - f * g.U;
        const bool live = f < g.phi && i < g.Ui;
        const int q0 = g.phi * i + f, P = g.P, Q = g.Q, nseg = g.nseg, qstep = g.phi * g.Ui;
        auto rows = [=](int64_t ti, int, int64_t& m) -> bool {
            const int T = t_lo + (int)ti;
            const int strip = T / P, p = T - strip * P;
            const int n = strip / nseg, q = (strip - n * nseg) * qstep + q0;
            m = ((int64_t)n * P + p) * Q + q;
            return live && q < Q;
        };
        ws_epilogue<EPI>(ep, thr, rows, t_hi - t_lo, n0, N, BN, sp, lacc, tmem_base, acc_scale, tfull, tempty,
                               err, warp, lane);
    }

    __syncthreads();
    if (*err && tid == 0) record_status(ep.status, ESB_ERR_TIMEOUT);
    if (warp == kWsMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

// ------------------------------------------------------------- host side

typedef void (*StemKernel)(StemGeom, const uint32_t*, int64_t, int64_t, OpFmt, OpFmt, int, int, int, int, float, EpiParams);
static const StemKernel kStemKernels[4] = {esb_conv_stem_kernel<kEpiB4>, esb_conv_stem_kernel<kEpiLean4>,
                                           esb_conv_stem_kernel<kEpiGen>, esb_conv_stem_kernel<kEpiTable>};

static int stem_static_smem(cudaError_t* err)
{
    static int v = -1;
    if (v < 0) {
        size_t m = 0;
        for (StemKernel k : kStemKernels) {
            cudaFuncAttributes a;
            *err = cudaFuncGetAttributes(&a, k);
            if (*err != cudaSuccess) return -1;
            if (a.sharedSizeBytes > m) m = a.sharedSizeBytes;
        }
        v = (int)m;
    }
    return v;
}

struct StemPlan {
    StemGeom g;
    int BN, nkb;
    int64_t smem;
};

// Whether this kernel finishes before the im2col kernel, by a model of both in
// microseconds: a fixed part (launch, prologue; here also the filters' decode,
// 0.9 us a pass of 288 chunks), and waves of tiles (one CTA per SM) times a
// tile's cost.  Both tiles are 128 rows, but here only `use` = Q /
// (128 nseg) of them are outputs, so a costly epilogue counts 1 / use times; the
// im2col kernel pays for each filter tap's word (another filter width: code by
// code) and a longer prologue, and takes narrower N-tiles where few row tiles
// leave SMs idle (resident_bn).  A tile's two roles overlap but for about a
// quarter of the shorter one.
// Measured, this kernel and im2col, 7x7/2 -> 64, 4-bit codes alone: 295 and 291
// us at 26 columns (use 0.2), 125 and 282 at 64, 85 and 286 at 100; with a
// scale per channel 592 and 381 at 64, 392 and 382 at 100; with y 847 and 327
// at 32; 2x2/2 -> 287, 3-bit, at 26: 283 and 69; 6-bit 3x3/2 -> 64: 134 and 101
// at 64, 91 and 101 at 100; one image of 224 x 224: 10.5 and 19.2; 10 x 10 -> 164
// sums alone, batch 3: 26.0 and 14.2; 11x11/2 -> 238, 6-bit, 11 x 13, batch 20: 52.2
// and 29.3.
static bool stem_pays(const StemGeom& g, int64_t n, int64_t N, int BN, int nkb, int out_cpw, bool mixed, double e16)
{
    const double sms = device_sm_count();
    const int64_t m = n * g.P * g.Q;
    const int bni = resident_bn(m, N, out_cpw, BN);
    const double epi = e16 * BN / 16, epi_i = e16 * bni / 16;
    const double gather = fmax(2.0, 0.5 + 0.15 * g.R * g.S) * (mixed ? 3 : 1);
    const double im2col = 14.0 + ceil((double)(((m + kBM - 1) / kBM) * ((N + bni - 1) / bni)) / sms) *
                                    (fmax(epi_i, gather) + 0.25 * fmin(epi_i, gather));
    const double filters = fmax(0.0, nkb * 8.0 * BN / (kWsProdWarp0 * 32) - 9.0);   // passes past the fixed part's
    const double stem = 9.0 + 0.9 * filters + ceil((double)(n * g.P * g.nseg * ((N + BN - 1) / BN)) / sms) * fmax(epi, 0.8 + 0.06 * g.R * g.G);
    return stem < im2col;
}

// Up to 4 channels, stride 2 or 4 (stride 1 has the halo kernel), whole-byte
// formats, where it pays (stem_pays).  e16: the epilogue's cost (epi_cost16).
static bool stem_plan(const esb_conv_desc& d, int P, int Q, int64_t ldx, int bx, int kx, int bw, int kw, int bn0, int out_cpw,
                      double e16, StemPlan* sp, cudaError_t* err)
{
    *err = cudaSuccess;
    if (d.c > 4 || (d.stride != 2 && d.stride != 4) || fmt_needs_split(bx, kx) || fmt_needs_split(bw, kw) || d.r > 16 || d.s > 16 ||
        ldx > (1 << 20) || bn0 <= 0)
        return false;
    StemGeom& g = sp->g;
    g.X = nullptr;
    g.ldx = (int)ldx; g.H = d.h; g.W = d.w; g.P = P; g.Q = Q; g.R = d.r; g.S = d.s; g.C = d.c; g.stride = d.stride; g.pad = d.pad;
    g.phi = 4 / d.stride;
    g.G = 2 * ((d.s + 7) / 8);
    const int per = (Q + g.phi - 1) / g.phi;                       // outputs of one residue in a row
    const int umax = kBM / g.phi;
    g.nseg = (per + umax - g.G) / (umax - g.G + 1);
    g.Ui = (per + g.nseg - 1) / g.nseg;
    g.U = g.Ui + g.G - 1;
    sp->BN = bn0;
    sp->nkb = (d.r * g.G * 16 + kBK - 1) / kBK;
    if ((int64_t)d.n * P * g.nseg >= (1ll << 30) || !stem_pays(g, d.n, d.cout, bn0, sp->nkb, out_cpw, bx != bw, e16)) return false;
    g.pitch = (kBM + g.G - 1) * 16;
    const int st = stem_static_smem(err);
    if (st < 0) return false;
    const int64_t maxs = max_dyn_smem() - st;
    const int64_t fixed = 1024 + (int64_t)sp->nkb * bn0 * kBK + 4 * 128 + (2 * kStemMaxRing + 2 * kMaxAcc + 1) * 8 + 64;
    int64_t nr = (maxs - fixed) / g.pitch;
    if (nr > kStemMaxRing) nr = kStemMaxRing;
    // a tile's rows and two more output rows' worth; a decoder's next row is within one turn of the ring
    if (nr < d.r + 2 * d.stride || nr < kWsProdWarps + 1) return false;
    g.NR = (int)nr;
    sp->smem = fixed + nr * g.pitch;
    return true;
}

bool conv_stem_ok(const esb_conv_desc& d, int P, int Q, int64_t ldx, int bx, int kx, int bw, int kw, int out_b)
{
    StemPlan sp;
    cudaError_t e;
    const int bn = pick_bn(d.cout, 32 / out_b);
    return bn > 0 && stem_plan(d, P, Q, ldx, bx, kx, bw, kw, bn, 32 / out_b, epi_cost16_codes(out_b), &sp, &e);
}

bool launch_conv_stem(const esb_conv_desc& d, int P, int Q, const uint32_t* X, int64_t ldx, const OpFmt& fa, const uint32_t* W,
                      int64_t ldw, const OpFmt& fb, int BN, const EpiParams& ep, cudaStream_t st, cudaError_t* err)
{
    StemPlan sp;
    if (!stem_plan(d, P, Q, ldx, fa.b, fa.k, fb.b, fb.k, BN, ep.out_cpw, epi_cost16(ep), &sp, err)) return *err != cudaSuccess;
    sp.g.X = X;
    static bool configured = false;
    if (!configured) {
        for (StemKernel k : kStemKernels) {
            *err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem() - stem_static_smem(err));
            if (*err != cudaSuccess) return true;
        }
        configured = true;
    }
    const int64_t N = d.cout;
    const int n_tiles = (int)((N + BN - 1) / BN);
    const int m_tiles = d.n * P * sp.g.nseg;
    int64_t per_n = device_sm_count() / n_tiles;
    if (per_n < 1) per_n = 1;
    if (per_n > m_tiles) per_n = m_tiles;
    const float acc_scale = ldexpf(1.0f, fa.csc + fb.csc);
    *err = launch_pdl(kStemKernels[epi_kind(ep)], dim3((unsigned)(per_n * n_tiles)), dim3(kWsThreads),
                      (size_t)sp.smem, st, sp.g, W, ldw, N, fa, fb, BN, sp.nkb, n_tiles, m_tiles, acc_scale, ep);
    return true;
}

}  // namespace esb
