// esb_conv_halo.cu -- stride-1 ESB convolution from a decoded input halo
// (Sec. IV-B: the r x s x c_in x c_out convolution of the computing logic).
//
// The im2col kernel (esb_gemm.cu) decodes every input code once per filter
// tap.  Here a 128-row output tile is rows_out = 128 / Ws whole output rows
// of one image, each padded to a pitch of Ws pixel slots (Ws = the power of
// two >= w + pad).  The producers decode the rows_out + r - 1 input rows
// that tile needs ONCE into shared memory, pixel-linear: slot
// (i * Ws + j + pad) holds input pixel (row p0 - pad + i, column j), and the
// slots of columns w .. Ws - 1, of the left padding and of rows outside the
// image hold E4M3 zero bytes (the decoded zero code).  Each 16-code channel
// chunk is its own plane of slots x 16 bytes.
//
// Output pixel (p0 + pl, q) is tile row pl * Ws + q, and its tap (r, s)
// reads slot (pl * Ws + q) + r * Ws + s.  So tap (r, s) of the whole tile is
// the same buffer seen from a start address shifted by (r * Ws + s) * 16
// bytes: with A in the K-major no-swizzle layout (rows 16 bytes apart in
// 8-row core matrices, SBO = 128 bytes between them, LBO = one plane between
// 16-code chunks), every tap is one descriptor, and the MMA warp issues
// r * s * (chunks / 2) tcgen05.mma (K = 32) per tile from a single decode.
// B (the filters, K = (tap, channel)) is resident, in the same layout: planes
// of BN rows x 16 bytes, BN * 16 + 16 bytes apart (the decoders' 8-lane stores
// then hit distinct banks), so that the descriptors of both operands advance
// by constants from one K step to the next.  The epilogue is the shared one; rows with q >= Q or past the image's last
// output row are computed from zero slots and not stored.
//
// Channel blocks of 128 codes are separate stages, so a tile's halo never
// needs more than 8 planes of shared memory at once.
#include <cstdint>
#include <cuda_runtime.h>

#include "esb_tc.cuh"

namespace esb {

constexpr int kHaloDecoders = kWsProdWarps - 1;   // bulk path: warps decoding each tile together

struct HaloGeom {
    const uint32_t* X;   // n*h*w pixels of ldx words
    int ldx;             // words per pixel (multiple of 4)
    int H, W, P, Q, R, S, pad;
    int lws;             // log2(Ws)
    int rows_out;        // output rows per tile (128 / Ws)
    int tpi;             // tiles per image
    int hr;              // halo rows (rows_out + R - 1)
    int ns;              // slots per plane (128 + (R-1) * Ws + S - 1)
    int pb;              // bytes per plane (ns * 16)
    int tail;            // pixels of the last input row: W, or fewer where a 1x1's pixels are taken 128 at a time
    int cblocks;         // channel blocks of 16 words
    int spw;             // K slots per input word: 8 (4-bit codes, 5/6-bit word slots) or 16 (2/3-bit word slots)
    int stage_bytes;     // planes of one channel block (<= 8 planes), then raw rows
    int planes_bytes;    // the planes part of a stage
    int raw_bytes;       // raw code rows of a tile (one channel block only), or 0: register path
};

// A CTA's tiles first, first + step, ... as (image, tile within it) without a
// division per tile (each role's scalar work per tile counts: its instructions
// come one per 5 to 10 cycles).
struct TileCursor {
    int img, t;
    int dimg, dt, tpi;
    __device__ __forceinline__ TileCursor(int first, int step, int tiles_per_image)
        : img(first / tiles_per_image), t(first - (first / tiles_per_image) * tiles_per_image), dimg(step / tiles_per_image),
          dt(step - (step / tiles_per_image) * tiles_per_image), tpi(tiles_per_image) {}
    __device__ __forceinline__ void next()
    {
        img += dimg;
        t += dt;
        if (t >= tpi) { t -= tpi; img++; }
    }
};

// The MMAs of one stage (channel block) with every offset a compile-time
// constant: slot pitch WS, an R x S filter, UT K steps of 32 codes per tap
// of which this block holds PAIRS, N-tile BN.  Straight-line issue, nothing
// but the tcgen05.mma between two MMAs.
template <int WS, int R, int S, int UT, int PAIRS, int BN>
__device__ __forceinline__ void halo_mma_fixed(uint32_t d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t& acc, uint32_t leader)
{
    constexpr int NS = 128 + (R - 1) * WS + S - 1;
    constexpr uint32_t PB = NS * 16;
#pragma unroll
    for (int t = 0; t < R * S; t++) {
#pragma unroll
        for (int j = 0; j < PAIRS; j++) {
            const uint32_t ao = (uint32_t)((((t / S) * WS + (t % S)) * 16 + 2 * j * (int)PB) >> 4);
            const uint32_t bo = (uint32_t)((t * UT + j) * 2 * (BN + 1));
            mma_f8f6f4(d, a_desc + ao, b_desc + bo, idesc, acc, leader);
            acc = 1u;
        }
    }
}

// One 4-word piece (piece pc of the pixel in slot `slot`) into its planes:
// 2 planes (pc * 2 ..) for 8-slot words, 4 planes (pc * 4 ..) for 16-slot
// words.  Pieces outside the image are zero codes.
template <int B>
__device__ __forceinline__ void halo_store_piece(uint8_t* st, int pb, int slot, int pc, const uint4& v, int k, int ew)
{
    constexpr int RW = SlotFmt<B>::SPW / 4;           // registers per word; planes per piece
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint8_t* dst = st + (RW * pc) * pb + slot * 16;
#pragma unroll
    for (int c = 0; c < RW; c++) {
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4 / RW; i++) decode_slots<B>(w[c * (4 / RW) + i], k, ew, o + i * RW);
        *reinterpret_cast<uint4*>(dst + c * pb) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// Item i of a stage fill is piece i % npc of slot i / npc (1 <= npc <= 4; i
// below 2^14: exact with a 16-bit reciprocal).
__device__ __forceinline__ int halo_slot(int i, int npc, uint32_t recip)
{
    return npc == 4 ? i >> 2 : (int)(((uint32_t)i * recip) >> 16);
}

// Register fills (several channel blocks): every producer thread takes
// kFillLoads pieces of a batch, so a batch is kWsProdWarps * 32 * kFillLoads
// items and a stage a few batches.  Filling each stage with all producer
// warps, rather than a stage per warp, keeps them all busy when only two
// stages fit beside the filters, and the next batch's loads are in flight
// while the current one is decoded.
constexpr int kFillLoads = 4;
constexpr int kFillBatch = kWsProdWarps * 32 * kFillLoads;

struct HaloCursor {                                   // a batch: tile, channel block, first item
    int64_t ti;
    int cb, i0;
};

// Geometry of a batch's stage: items, pieces per slot.
__device__ __forceinline__ int halo_npc(const HaloGeom& g, int cb) { return min(16, g.ldx - cb * 16) >> 2; }

__device__ __forceinline__ void halo_load(const HaloGeom& g, int T, int cb, int i0, int t, uint32_t zw, uint4 (&v)[kFillLoads])
{
    const int nimg = T / g.tpi;
    const int p0 = (T - nimg * g.tpi) * g.rows_out;
    const int npc = halo_npc(g, cb);
    const uint32_t recip = 65536u / (uint32_t)npc + 1u;
    const int wsm = (1 << g.lws) - 1;
    const uint32_t* xi = g.X + (int64_t)nimg * g.H * g.W * g.ldx + cb * 16;
#pragma unroll
    for (int u = 0; u < kFillLoads; u++) {
        const int i = i0 + u * kWsProdWarps * 32 + t;
        const int slot = halo_slot(i, npc, recip), pc = i - slot * npc;
        const int rel = slot - g.pad;
        const int hi = rel >> g.lws;                               // halo row (-1: left guard)
        const int j = rel & wsm;
        const int h = p0 - g.pad + hi;
        const bool ok = slot < g.ns && rel >= 0 && hi < g.hr && (unsigned)h < (unsigned)g.H && j < (h + 1 < g.H ? g.W : g.tail);
        v[u] = make_uint4(zw, zw, zw, zw);
        if (ok) v[u] = __ldg(reinterpret_cast<const uint4*>(xi + ((int64_t)h * g.W + j) * g.ldx) + pc);
    }
}

template <int B>
__device__ __forceinline__ void halo_store(const HaloGeom& g, int cb, int i0, int t, uint8_t* st, const uint4 (&v)[kFillLoads],
                                           int k, int ew)
{
    const int npc = halo_npc(g, cb);
    const uint32_t recip = 65536u / (uint32_t)npc + 1u;
#pragma unroll
    for (int u = 0; u < kFillLoads; u++) {
        const int i = i0 + u * kWsProdWarps * 32 + t;
        const int slot = halo_slot(i, npc, recip);
        if (slot < g.ns) halo_store_piece<B>(st, g.pb, slot, i - slot * npc, v[u], k, ew);
    }
}

// Bulk-copy fills (one channel block, ldx <= 16 words).  The copy issuer
// (one thread) copies the input rows of tile T that lie inside the image,
// whole (w pixels of ldx words, contiguous in NHWC), into the stage's raw
// area with one cp.async.bulk each, completing on mbarrier `raw_bar`.
__device__ __forceinline__ void halo_issue_rows(const HaloGeom& g, int nimg, int p0, uint8_t* st, uint64_t* raw_bar)
{
    uint8_t* raw = st + g.planes_bytes;
    const uint32_t row_bytes = (uint32_t)(g.W * g.ldx) * 4u;
    const int h0 = p0 - g.pad;
    const int lo = h0 < 0 ? -h0 : 0;                               // rows lo .. hi - 1 lie in the image
    const int hi = g.H - h0 < g.hr ? g.H - h0 : g.hr;
    const uint32_t last = (uint32_t)(g.tail * g.ldx) * 4u;
    const bool cut = h0 + hi == g.H;                               // the image's last row is among them
    uint32_t bytes = hi > lo ? (uint32_t)(hi - lo) * row_bytes : 0u;
    if (cut && hi > lo) bytes -= row_bytes - last;
    mbar_arrive_expect_tx(raw_bar, bytes);
    const uint32_t* src = g.X + ((int64_t)nimg * g.H + h0 + lo) * (int64_t)(g.W * g.ldx);
    for (int i = lo; i < hi; i++, src += g.W * g.ldx)
        bulk_copy_g2s(raw + (size_t)i * row_bytes, src, cut && i + 1 == hi ? last : row_bytes, raw_bar);
}

// The decoders' share of one bulk-filled tile: items first, first + stride,
// ... (zero codes for padding slots and rows outside the image).
template <int B>
__device__ __forceinline__ void halo_decode(const HaloGeom& g, int p0, uint8_t* st, int first, int stride, int k, int ew,
                                            uint32_t zw)
{
    const uint8_t* raw = st + g.planes_bytes;
    const int wsm = (1 << g.lws) - 1;
    const int npc = g.ldx >> 2;
    const uint32_t recip = 65536u / (uint32_t)npc + 1u;
    const int items = g.ns * npc;
#pragma unroll 1                                      // compact: it shares the SM's instruction cache
    for (int i = first; i < items; i += stride) {
        const int slot = halo_slot(i, npc, recip), pc = i - slot * npc;
        const int rel = slot - g.pad;
        const int hi = rel >> g.lws;
        const int j = rel & wsm;
        const int h = p0 - g.pad + hi;
        const bool ok = rel >= 0 && hi < g.hr && (unsigned)h < (unsigned)g.H && j < (h + 1 < g.H ? g.W : g.tail);
        const uint4* src = reinterpret_cast<const uint4*>(raw + ((size_t)hi * g.W + j) * g.ldx * 4);
        halo_store_piece<B>(st, g.pb, slot, pc, ok ? src[pc] : make_uint4(zw, zw, zw, zw), k, ew);
    }
}

// The same out of line, for the instances that hold every width.
template <int B>
__device__ __noinline__ void halo_decode_call(const HaloGeom g, int T, uint8_t* st, int first, int stride, int k, int ew)
{
    const int nimg = T / g.tpi;
    halo_decode<B>(g, (T - nimg * g.tpi) * g.rows_out, st, first, stride, k, ew, fmt_zero_word(B, k));
}

template <bool FAST, int EPI>
__global__ void __launch_bounds__(kWsThreads, 1)
esb_conv_halo_kernel(HaloGeom g, RowsSrc srcB, int64_t N, int64_t K, OpFmt fa, OpFmt fb, int BN, int nkb,
                     int stages, int n_tiles, int64_t m_tiles, float acc_scale, const __grid_constant__ EpiParams ep)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int b_pitch = (BN + 1) * 16;                         // chunk planes of B
    uint8_t* sB = smem;                                        // 8 nkb planes
    uint8_t* sA = sB + nkb * 8 * b_pitch;                      // stages x stage_bytes (halo planes), 128-byte aligned
    float* thr = reinterpret_cast<float*>(sA + stages * g.stage_bytes);
    uint64_t* full = reinterpret_cast<uint64_t*>(thr + 128);
    uint64_t* empty = full + kWsMaxStages;
    uint64_t* tfull = empty + kWsMaxStages;
    uint64_t* tempty = tfull + kMaxAcc;
    uint64_t* drain = tempty + kMaxAcc;
    uint64_t* rawb = drain + 1;                                // kWsMaxStages: bulk-copy fills
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(rawb + kWsMaxStages);
    volatile int* err = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x;
    const int warp = warp_index(), lane = tid & 31;
    const int n_tile = (int)(blockIdx.x % n_tiles);
    const int64_t cta_in_n = blockIdx.x / n_tiles;
    const int64_t ctas_per_n = gridDim.x / n_tiles;
    const int64_t n0 = (int64_t)n_tile * BN;
    const int64_t my_tiles = (m_tiles > cta_in_n) ? (m_tiles - cta_in_n + ctas_per_n - 1) / ctas_per_n : 0;
    const int lacc = acc_buffers_log2(BN);
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < (BN << lacc)) tmem_cols <<= 1;
    const EpiSplit sp = epi_split<EPI>(ep, BN, my_tiles);
    const int cbs = g.cblocks;
    // the layout above must fit the dynamic allocation (uniform for the CTA)
    if ((uintptr_t)(reinterpret_cast<const volatile uint8_t*>(err) + 4 - smem_raw) > dynamic_smem_bytes()) {
        if (tid == 0) record_status(ep.status, ESB_ERR_INTERNAL);
        return;
    }

    {
        // the CTA's rows of B into L2 while the previous grid may still be
        // finishing (weights are often no longer in L2 by the next call)
        const int64_t rows_b = (srcB.rows - n0) < (int64_t)BN ? (srcB.rows - n0) : (int64_t)BN;
        const char* b0 = reinterpret_cast<const char*>(srcB.base + n0 * srcB.ld);
        const int64_t bytes = rows_b > 0 ? rows_b * srcB.ld * 4 : 0;
        for (int64_t off = (int64_t)tid * 128; off < bytes; off += (int64_t)kWsThreads * 128) prefetch_l2(b0 + off);
    }
    if (tid == 0) {
        for (int s = 0; s < stages; s++) {
            // the decoder warps (register path: every producer warp) fill a stage together
            mbar_init(&full[s], g.raw_bytes > 0 ? kHaloDecoders : kWsProdWarps);
            mbar_init(&empty[s], 1);
            mbar_init(&rawb[s], 1);                   // the issuer's arrive.expect_tx, then the copies' bytes
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
    griddep_wait();                                   // X, B and the alphas may come from the previous launch
    griddep_launch_dependents();                      // every CTA is resident: the next grid may queue behind it

    // Setup.  Every warp but the bulk issuer (which starts the first tiles'
    // row copies at once) decodes its share of B, one row chunk per thread
    // where it can, so that B is ready after about one load round trip; the
    // MMA warp waits for all of it on named barrier 1, the others only
    // arrive.  The epilogue warps then build the requantisation thresholds
    // (named barrier 3) while the first tile is filled and multiplied.
    const bool bulk = FAST || g.raw_bytes > 0;
    if (!(bulk && warp == kWsProdWarp0)) {
        const int nbdec = bulk ? kWsThreads - 32 : kWsThreads;
        const int t = (bulk && warp > kWsProdWarp0) ? tid - 32 : tid;
        ws_decode_b<FAST>(srcB, n0, K, fb, BN, nkb, sB, t, nbdec, nullptr, b_pitch);
        fence_proxy_async_smem();
        if (warp == kWsMmaWarp) asm volatile("bar.sync 1, %0;" ::"r"(nbdec) : "memory");
        else asm volatile("bar.arrive 1, %0;" ::"r"(nbdec) : "memory");
    }
    if (warp < kWsEpiWarps) ws_thresholds(thr, ep, warp, lane);
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp >= kWsProdWarp0) {
        // ---------------------------------------------- halo producers
        const int p = warp - kWsProdWarp0;
        if (bulk) {
            // Bulk path, tiles in order: producer warp 0 issues the row copies
            // of every tile as soon as its stage is free (up to `stages` tiles
            // ahead); the other kHaloDecoders warps decode each tile together,
            // so the first tile is ready after one copy and a short decode.
            int s = 0;
            uint32_t ph = 0u;
            if (p == 0) {
                if (lane == 0) {
                    TileCursor tc((int)cta_in_n, (int)ctas_per_n, g.tpi);
                    for (int64_t ti = 0; ti < my_tiles && !*err; ti++, tc.next()) {
                        if (!wait_or_abort(&empty[s], ph ^ 1u, err)) { *err = 1; break; }
                        halo_issue_rows(g, tc.img, tc.t * g.rows_out, sA + s * g.stage_bytes, &rawb[s]);
                        if (++s == stages) { s = 0; ph ^= 1u; }
                    }
                }
            } else {
                const int d = p - 1;                  // decoder index 0 .. kHaloDecoders - 1
                auto decode_tiles = [&](auto width) {
                    constexpr int B = decltype(width)::value;
                    TileCursor tc((int)cta_in_n, (int)ctas_per_n, g.tpi);
                    const uint32_t zw = fmt_zero_word(B, fa.k);
                    for (int64_t ti = 0; ti < my_tiles && !*err; ti++) {
                        if (!wait_or_abort(&rawb[s], ph, err)) { *err = 1; break; }
                        uint8_t* const st = sA + s * g.stage_bytes;
                        if (FAST) {
                            halo_decode<B>(g, tc.t * g.rows_out, st, d * 32 + lane, kHaloDecoders * 32, fa.k, fa.ew, zw);
                            tc.next();
                        } else {
                            halo_decode_call<B>(g, (int)(cta_in_n + ti * ctas_per_n), st, d * 32 + lane, kHaloDecoders * 32, fa.k,
                                                fa.ew);
                        }
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[s]);
                        if (++s == stages) { s = 0; ph ^= 1u; }
                    }
                };
                if (FAST) decode_tiles(IntC<4>());
                else with_width(fa.b, decode_tiles);
            }
        } else if constexpr (!FAST) {
            // Register path (several channel blocks): the (tile, channel
            // block) stages in order, each filled by every producer warp.
            const int t = p * 32 + lane;
            with_width(fa.b, [&](auto width) {
                constexpr int B = decltype(width)::value;
                const uint32_t zw = fmt_zero_word(B, fa.k);
                uint4 v[kFillLoads];
                HaloCursor c{0, 0, 0};
                int s = 0;
                uint32_t ph = 0u;
                if (my_tiles > 0) halo_load(g, (int)cta_in_n, 0, 0, t, zw, v);
                while (c.ti < my_tiles && !*err) {
                    if (c.i0 == 0 && !wait_or_abort(&empty[s], ph ^ 1u, err)) { *err = 1; break; }
                    // the next batch: the same stage's rest, else the next stage's start
                    HaloCursor nx = c;
                    nx.i0 += kFillBatch;
                    const bool last = nx.i0 >= g.ns * halo_npc(g, c.cb);
                    if (last) {
                        nx.i0 = 0;
                        if (++nx.cb == cbs) { nx.cb = 0; nx.ti++; }
                    }
                    uint4 vn[kFillLoads];
                    if (nx.ti < my_tiles) halo_load(g, (int)(cta_in_n + nx.ti * ctas_per_n), nx.cb, nx.i0, t, zw, vn);
                    halo_store<B>(g, c.cb, c.i0, t, sA + s * g.stage_bytes, v, fa.k, fa.ew);
                    if (last) {
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[s]);
                        if (++s == stages) { s = 0; ph ^= 1u; }
                    }
#pragma unroll
                    for (int u = 0; u < kFillLoads; u++) v[u] = vn[u];
                    c = nx;
                }
            });
        }
    } else if (warp == kWsMmaWarp) {
        // ---------------------------------------------- MMA issue
        // Common geometries issue straight-line MMAs with constant offsets
        // (halo_mma_fixed); others compute the offsets in the loop.
        // Descriptors never come from shared memory: the tensor core's own
        // operand reads keep it close to saturated.
        const uint32_t idesc = idesc_e4m3_f32(BN);
        const uint32_t leader = elect_one();
        const int ws = 1 << g.lws;
        const int units_tap = (g.ldx * g.spw) >> 5;            // 32-slot K steps per tap
        const bool r3 = g.R == 3 && g.S == 3;
        const uint64_t a_desc = smem_desc_noswz(smem_u32(sA), (uint32_t)g.pb, 128u);
        const uint64_t b_desc = smem_desc_noswz(smem_u32(sB), (uint32_t)b_pitch, 128u);
        // in the descriptors' 16-byte units
        const uint64_t a_step = (uint64_t)(g.stage_bytes >> 4), p_step = (uint64_t)((2 * g.pb) >> 4);
        const uint64_t b_step = (uint64_t)((2 * b_pitch) >> 4);
        int s = 0;                                             // stage and phase of the next K-block
        uint32_t ph = 0u;
        bool ok = true;
        for (int64_t ti = 0; ti < my_tiles && ok; ti++) {
            const int a = (int)(ti & ((1 << lacc) - 1));
            ok = warp_wait(&tempty[a], (uint32_t)((ti >> lacc) & 1) ^ 1u, err);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d = tmem_base + (uint32_t)(a * BN);
            uint32_t acc = 0u;
            for (int cb = 0; cb < cbs; cb++) {
                ok = warp_wait(&full[s], ph, err);
                if (!ok) break;
                tc_fence_after();
                const uint64_t a_st = a_desc + (uint64_t)s * a_step;
                const uint64_t b_blk = b_desc + (uint64_t)(cb * (g.spw >> 1)) * b_step;   // block cb: 16 words on
                const int pairs = (min(16, g.ldx - cb * 16) * g.spw) >> 5;   // K steps (plane pairs) of the block
                if (r3 && ws == 64 && units_tap == 2 && BN == 64) {           // 56 x 56 x 64
                    halo_mma_fixed<64, 3, 3, 2, 2, 64>(d, a_st, b_blk, idesc, acc, leader);
                } else if (r3 && ws == 32 && units_tap == 4 && BN == 128) {   // 28 x 28 x 128
                    halo_mma_fixed<32, 3, 3, 4, 4, 128>(d, a_st, b_blk, idesc, acc, leader);
                } else if (r3 && ws == 16 && units_tap == 8 && pairs == 4 && BN == 64) {   // 14 x 14 x 256
                    halo_mma_fixed<16, 3, 3, 8, 4, 64>(d, a_st, b_blk, idesc, acc, leader);
                } else {
                    uint64_t bt0 = b_blk;
                    for (int r = 0; r < g.R; r++) {
                        for (int sx = 0; sx < g.S; sx++, bt0 += (uint64_t)units_tap * b_step) {
                            uint64_t at = a_st + (uint64_t)(r * ws + sx), bt = bt0;
#pragma unroll 4
                            for (int j = 0; j < pairs; j++, at += p_step, bt += b_step) {
                                mma_f8f6f4(d, at, bt, idesc, acc, leader);
                                acc = 1u;
                            }
                        }
                    }
                }
                mma_commit(&empty[s], leader);
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
            if (ok) mma_commit(&tfull[a], leader);
        }
        if (!ok) *err = 1;
        ws_drain(drain, err, leader);
    } else if (warp < sp.warps) {
        // ---------------------------------------------- epilogue
        // tile counts fit in 32 bits (host check)
        const int rows_out = g.rows_out, lws = g.lws, P = g.P, Q = g.Q, tpi = g.tpi;
        const int qlast = g.tail < g.W ? g.tail : Q;              // outputs of the last row
        const int ctas = (int)ctas_per_n, first = (int)cta_in_n;
        auto rows = [=](int64_t ti, int row, int64_t& m) -> bool {
            const int T = first + (int)ti * ctas;
            const int nimg = T / tpi;
            const int p = (T - nimg * tpi) * rows_out + (row >> lws);
            const int q = row & ((1 << lws) - 1);
            m = ((int64_t)nimg * P + p) * Q + q;
            return p < P && q < (p + 1 < P ? Q : qlast);
        };
        ws_epilogue<EPI>(ep, thr, rows, my_tiles, n0, N, BN, sp, lacc, tmem_base, acc_scale, tfull, tempty, err,
                    warp, lane);
    }

    __syncthreads();
    if (*err && tid == 0) record_status(ep.status, ESB_ERR_TIMEOUT);
    if (warp == kWsMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

// Minimum share of the computed tile rows that are real output pixels for
// the halo path to be taken (56 x 56: 87.5 %; 7 x 7: 38 %, im2col instead).
constexpr double kHaloMinUse = 0.7;

struct HaloPlan {
    HaloGeom g;
    int BN, nkb, stages;
    int64_t K, smem, tiles;
};

// The instances by epilogue (epi_kind); [kEpiLean4] is the specialised one: 4-bit
// B, bulk-copied input rows.
typedef void (*HaloKernel)(HaloGeom, RowsSrc, int64_t, int64_t, OpFmt, OpFmt, int, int, int, int, int64_t, float, EpiParams);
static const HaloKernel kHaloKernels[4] = {esb_conv_halo_kernel<false, kEpiB4>, esb_conv_halo_kernel<true, kEpiLean4>,
                                           esb_conv_halo_kernel<false, kEpiGen>, esb_conv_halo_kernel<false, kEpiTable>};

// Static shared memory of the kernel (the largest of its instances).
static int halo_static_smem(cudaError_t* err)
{
    static int v = -1;
    if (v < 0) {
        size_t m = 0;
        for (HaloKernel k : kHaloKernels) {
            cudaFuncAttributes a;
            *err = cudaFuncGetAttributes(&a, k);
            if (*err != cudaSuccess) return -1;
            if (a.sharedSizeBytes > m) m = a.sharedSizeBytes;
        }
        v = (int)m;
    }
    return v;
}

// Geometry, N-tile width and shared-memory budget of the halo path, or
// false when the shape does not suit it.  BN starts at bn0 and shrinks
// (keeping whole output words) until the resident B and two halo stages fit.
// e16: the epilogue's cost (epi_cost16).
static bool halo_plan(const esb_conv_desc& d0, int P, int Q, int64_t ldx, const OpFmt& fa, int bn0, int out_cpw, double e16,
                      HaloPlan* hp, cudaError_t* err)
{
    *err = cudaSuccess;
    // A 1x1 filter sees no rows: its pixels are one image of rows of 128, so
    // that every tile is full whatever the width.  With one channel block only:
    // over several, image rows measured faster (28x28x144 -> 32: 12.0 against
    // 13.6 us; 7x7x960 -> 160 on the im2col kernel 16 against 23 us), while
    // 112x112x32 -> 16 gains 58 -> 48 us and 56x56x24 -> 144 33 -> 30.  Not where
    // a costly epilogue meets fewer tiles than SMs: the im2col kernel then takes
    // narrower N-tiles (66x68x64 -> 97, batch 2, 8-bit codes with a residual: 53.4
    // us here, 24.0 there).
    esb_conv_desc d = d0;
    hp->g.tail = d.w;
    const int64_t pixels = (int64_t)d.n * d.h * d.w;
    const bool idle = bn0 > 0 && (pixels + kBM - 1) / kBM * ((d.cout + bn0 - 1) / bn0) < device_sm_count();
    if (d.r == 1 && d.s == 1 && d.stride == 1 && d.pad == 0 && ldx <= 16 && !(idle && e16 >= 1.0)) {
        if (pixels >= (1ll << 30)) return false;
        d.n = 1;
        d.w = kBM;
        d.h = (int)((pixels + kBM - 1) / kBM);
        P = d.h;
        Q = kBM;
        hp->g.tail = (int)(pixels - (int64_t)(d.h - 1) * kBM);
    }
    hp->tiles = 0;
    // 4-bit codes, or 5/6-bit codes in the word-slot layout (8 K slots per
    // word, the same K per pixel word as 4-bit codes)
    const bool slot8 = fa.spw == 8 && (fa.b == 5 || fa.b == 6);
    const bool slot16 = fa.spw == 16 && (fa.b == 2 || fa.b == 3);
    if (d.stride != 1 || !(fa.b == 4 || slot8 || slot16) || fa.planes != 1 || ldx % 4 != 0 || ldx > (1 << 20) ||
        d.pad > d.r - 1 || d.pad > d.s - 1)
        return false;
    int lws = 0;
    while ((1 << lws) < d.w + d.pad) lws++;
    const int ws = 1 << lws;
    if (ws > kBM || Q > ws) return false;
    HaloGeom& g = hp->g;
    g.X = nullptr; g.ldx = (int)ldx; g.H = d.h; g.W = d.w; g.P = P; g.Q = Q; g.R = d.r; g.S = d.s; g.pad = d.pad;
    g.lws = lws;
    g.rows_out = kBM / ws;
    g.tpi = (P + g.rows_out - 1) / g.rows_out;
    if ((double)P * Q / ((double)g.tpi * kBM) < kHaloMinUse) return false;
    g.hr = g.rows_out + d.r - 1;
    g.ns = kBM + (d.r - 1) * ws + d.s - 1;
    g.pb = g.ns * 16;
    g.cblocks = (int)((ldx + 15) / 16);
    g.spw = slot16 ? 16 : 8;
    const int planes = (int)((ldx >= 16 ? 16 : ldx) * g.spw / 16);      // planes of one channel block
    g.planes_bytes = ((planes * g.pb + 127) / 128) * 128;
    // one channel block: the fill bulk-copies whole input rows to a raw area of the stage
    g.raw_bytes = (g.cblocks == 1) ? ((g.hr * d.w * (int)ldx * 4 + 127) / 128) * 128 : 0;
    g.stage_bytes = g.planes_bytes + g.raw_bytes;
    if ((int64_t)d.n * g.tpi >= (1ll << 30)) return false;
    hp->tiles = (int64_t)d.n * g.tpi;
    const int st_smem = halo_static_smem(err);
    if (st_smem < 0) return false;
    const int maxs = max_dyn_smem() - st_smem;
    hp->K = (int64_t)d.r * d.s * ldx * g.spw;
    hp->nkb = (int)((hp->K + kBK - 1) / kBK);
    static const int cands[] = {256, 240, 224, 208, 192, 176, 160, 144, 128, 112, 96, 80, 64, 48, 32, 16};
    for (int i = -1; i < (int)(sizeof(cands) / sizeof(cands[0])); i++) {
        const int bn = i < 0 ? bn0 : cands[i];
        if (bn <= 0 || (i >= 0 && bn >= bn0) || bn % out_cpw != 0) continue;
        const int64_t fixed = 1024 + (int64_t)hp->nkb * 8 * (bn + 1) * 16 + 4 * 128 + 512;
        int64_t stg = (maxs - fixed) / g.stage_bytes;
        if (stg > kWsMaxStages) stg = kWsMaxStages;
        if (stg < 2) continue;
        hp->BN = bn;
        hp->stages = (int)stg;
        hp->smem = fixed + stg * (int64_t)g.stage_bytes;
        return true;
    }
    return false;
}

bool conv_halo_ok(const esb_conv_desc& d, int P, int Q, int64_t ldx, int bx, int kx, int out_b)
{
    const int out_cpw = 32 / out_b;
    HaloPlan hp;
    cudaError_t e;
    OpFmt fa = make_opfmt(bx, kx);
    if (bx == 5 || bx == 6) fa.spw = 8;               // as plan_slots for same-width input and filters
    if (bx == 2 || bx == 3) fa.spw = 16;
    return halo_plan(d, P, Q, ldx, fa, pick_bn(d.cout, out_cpw), out_cpw, epi_cost16_codes(out_b), &hp, &e);
}

bool launch_conv_halo(const esb_conv_desc& d, int P, int Q, const uint32_t* X, int64_t ldx, const OpFmt& fa,
                      const uint32_t* W, int64_t ldw, const OpFmt& fb, int BN, const EpiParams& ep, cudaStream_t st,
                      cudaError_t* err)
{
    HaloPlan hp;
    if (!halo_plan(d, P, Q, ldx, fa, BN, ep.out_cpw, epi_cost16(ep), &hp, err)) return *err != cudaSuccess;
    if (hp.smem <= 0 || hp.smem > max_dyn_smem() - halo_static_smem(err)) {
        *err = cudaErrorInvalidConfiguration;
        return true;
    }
    hp.g.X = X;
    static bool configured = false;
    if (!configured) {
        for (HaloKernel k : kHaloKernels) {
            *err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem() - halo_static_smem(err));
            if (*err != cudaSuccess) return true;
        }
        configured = true;
    }
    const int64_t N = d.cout;
    const int n_tiles = (int)((N + hp.BN - 1) / hp.BN);
    const int64_t m_tiles = hp.tiles;
    int64_t per_n = device_sm_count() / n_tiles;
    if (per_n < 1) per_n = 1;
    if (per_n > m_tiles) per_n = m_tiles;
    const int64_t grid = per_n * n_tiles;
    RowsSrc b{W, (int64_t)d.r * d.s * ldw, N};
    const float acc_scale = ldexpf(1.0f, fa.csc + fb.csc);
    const int kind = epi_kind(ep);
    const bool fast = kind == kEpiLean4 && fb.b == 4 && hp.g.raw_bytes > 0;   // what the specialised instance takes
    *err = launch_pdl(kHaloKernels[kind == kEpiLean4 && !fast ? kEpiB4 : kind],
                      dim3((unsigned)grid), dim3(kWsThreads), (size_t)hp.smem, st, hp.g, b, N,
                      hp.K, fa, fb, hp.BN, hp.nkb, hp.stages, n_tiles, m_tiles, acc_scale, ep);
    return true;
}

}  // namespace esb
