// ESB GEMM for large operands (Sec. III-B products, Sec. IV-B/IV-C
// computing logic): C[m, n] = sum_k I(A[m, k]) I(B[n, k]) with the fused
// epilogue, for shapes whose B does not stay resident in shared memory.
//
// Two steps on the caller's stream:
//  1. esb_tile_kernel decodes each operand once into an image of E4M3 bytes
//     in the caller's workspace: K-block kb (128 codes) of row r at byte
//     (kb * rpad + r) * 128, its 16-byte chunk g at ((g ^ (r & 7)) * 16), so
//     any run of rows that starts at a multiple of 8 is one contiguous block
//     in the SW128 K-major layout of an MMA operand.  Rows past the operand
//     and codes past K are E4M3 zeros.  HBM-bound: code bytes in, one byte
//     per code out.
//  2. esb_gemm_tiled_kernel, persistent and warp-specialised: one producer
//     thread bulk-copies whole tiles (A: 128 rows, 16 KiB; B: BN rows,
//     up to 32 KiB) into a ring of shared-memory stages (cp.async.bulk
//     completing on mbarriers), the MMA thread issues four 128 x BN x 32
//     tcgen05.mma per K-block into one of two BN-column TMEM accumulators,
//     and eight epilogue warps drain them through the epilogue of the other
//     tcgen05 kernels (ws_epilogue).  Each CTA keeps one N-tile and walks
//     the M-tiles.  BN is at most 256, or 240 for outputs of 3, 5 or 6 bits,
//     whose 10, 6 or 5 codes per word divide 240 (a word never straddles
//     tiles), and down to 64 where few row tiles leave SMs idle (tiled_bn).
//     Measured at 4096^3 with 6-bit codes: 62 us for the call, against 1458
//     us for the streamed kernel, which decodes every operand row again in
//     each tile (the only one to take these widths before).
// The contraction is exact: fp32 TMEM accumulation of integer-valued
// products holds every partial sum exactly while it stays below 2^24, so a K
// with K max|I_A| max|I_B| >= 2^24 is split into chunks that each stay
// below it, accumulated in separate TMEM regions (up to four, with a
// 128-column N-tile beyond two) and added as integers in the epilogue
// (int32: K max|I_A| max|I_B| < 2^31).
#include <cstdint>
#include <cstdlib>
#include <cuda_runtime.h>

#include "esb_tc.cuh"
#include "esb_internal.h"

namespace esb {

namespace {

constexpr int kTiledBN = 256;                  // N-tile width (rows of a B tile); 128 with > 2 K-chunks
constexpr int kTiledBNOdd = 240;               // for 10, 6 or 5 output codes per word (3, 5, 6 bits)
constexpr int kTiledThreads = 320;             // warps 0-7 epilogue, 8 MMA, 9 producer
constexpr int kTiledProdWarp = 9;
constexpr int kTileA = kBM * kBK;              // 16 KiB
constexpr int kTmemCols = 512;

}  // namespace

// The 16-code unit [k0, k0 + 16) of a row as 16 E4M3 bytes in unit_pos order
// (any width, by a walk of its words: a code never straddles two words, one
// load per word), zeros past K.
__device__ __noinline__ uint4 tile_unit_any(const uint32_t* p, int64_t k0, int64_t K, const OpFmt f)
{
    uint32_t ob[4] = {0u, 0u, 0u, 0u};
    if (k0 < K) {
        int64_t wi = k0 / f.cpw;
        int slot = (int)(k0 - wi * f.cpw);
        uint32_t w = __ldg(p + wi);
#pragma unroll
        for (int j = 0; j < 16; j++) {
            if (k0 + j >= K) break;
            const uint32_t byte = code_to_e4m3((w >> (f.b * slot)) & f.mask, f);
            const int pos = unit_pos(j);
            ob[pos >> 2] |= byte << (8 * (pos & 3));
            if (++slot == f.cpw) {
                slot = 0;
                ++wi;
                if (k0 + j + 1 < K) w = __ldg(p + wi);
            }
        }
    }
    return make_uint4(ob[0], ob[1], ob[2], ob[3]);
}

// One operand of the tile pass.
struct TileSrc {
    const uint32_t* base;
    int64_t ld;
    int64_t rows;              // rows of the operand
    int64_t rpad;              // rows of the image: a multiple of 16, zeros past `rows`
    OpFmt f;
    int packed;                // both operands of the same 3-, 5- or 6-bit width: packed runs (tile_run)
    int64_t units;             // threads' units of work
    int upr;                   // units per row (packed)
    uint8_t* out;
};

// 16-byte chunk c of row r in the image: K-block c / 8, swizzled chunk c % 8.
__device__ __forceinline__ uint4* tile_chunk(const TileSrc& t, int64_t r, int c)
{
    return reinterpret_cast<uint4*>(t.out + ((int64_t)(c >> 3) * t.rpad + r) * kBK + (((c & 7) ^ (int)(r & 7)) << 4));
}

// 3/5/6-bit codes packed without gaps: a run of RW words whose codes are a
// whole number of 16-byte chunks (6-bit: 16 words = 80 codes = 5 chunks;
// 5-bit: 8 words = 48 codes = 3 chunks; 3-bit: 8 words = 80 codes = 5
// chunks).  The first 4 (3-bit: 8) codes of every word fill the run's first
// chunks, the 1 or 2 codes left over of all its words the last one.  The
// same K order on both operands, so the sums are those of any other order;
// about 3.5 instructions per code (the per-code walk takes 12).
template <int B>
struct TileRun {
    static constexpr int CPW = 32 / B;
    static constexpr int RW = B == 6 ? 16 : 8;
    static constexpr int CODES = RW * CPW;
    static constexpr int CHUNKS = CODES / 16;
};

template <int B>
__device__ __forceinline__ void tile_run(const TileSrc& t, int64_t r, const uint32_t* p, int run)
{
    constexpr int RW = TileRun<B>::RW, CH = TileRun<B>::CHUNKS;
    uint32_t w[RW];
    const uint4* q = reinterpret_cast<const uint4*>(p + (int64_t)run * RW);   // rows are 16-byte aligned
#pragma unroll
    for (int i = 0; i < RW / 4; i++) {
        const uint4 v = __ldg(q + i);
        w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
    }
    const int k = t.f.k;
    const int c0 = run * CH;
#pragma unroll
    for (int i = 0; i < RW; i++) w[i] = rot_word<B>(w[i], k);
    uint32_t rest[4] = {0u, 0u, 0u, 0u};              // the last chunk's bytes: fields still at their low bits
#pragma unroll
    for (int c = 0; c + 1 < CH; c++) {
        uint32_t o[4];
        if (B == 3) {
#pragma unroll
            for (int i = 0; i < 2; i++) {
                o[2 * i] = e4m3_4<B>(spread4<B>(w[2 * c + i]), k);
                o[2 * i + 1] = e4m3_4<B>(spread4<B>(w[2 * c + i] >> 12), k);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; i++) o[i] = e4m3_4<B>(spread4<B>(w[4 * c + i]), k);
        }
        *tile_chunk(t, r, c0 + c) = make_uint4(o[0], o[1], o[2], o[3]);
    }
#pragma unroll
    for (int i = 0; i < RW; i++) {
        if (B == 6) {
            rest[i >> 2] |= ((w[i] >> 24) & 0x3fu) << (8 * (i & 3));
        } else {
            constexpr int SH = B == 5 ? 20 : 24;      // the word's last two codes
            constexpr uint32_t CM = (1u << B) - 1u;
            const uint32_t g = w[i] >> SH;
            rest[i >> 1] |= ((g & CM) | ((g << (8 - B)) & (CM << 8))) << (16 * (i & 1));
        }
    }
#pragma unroll
    for (int i = 0; i < 4; i++) rest[i] = e4m3_4<B>(rest[i], k);
    *tile_chunk(t, r, c0 + CH - 1) = make_uint4(rest[0], rest[1], rest[2], rest[3]);
}

// Unit u of a packed operand: run u % upr of row u / upr; the last unit of a
// row is its tail (the codes past the whole runs, then zeros to the end of
// the last K-block), by the per-code walk.
template <int B>
__device__ __forceinline__ void tile_packed(const TileSrc& t, int64_t u, int64_t K, int nkb)
{
    const int64_t r = u < (1ll << 32) ? (int64_t)((uint32_t)u / (uint32_t)t.upr) : u / t.upr;
    const int run = (int)(u - r * t.upr);
    const bool live = r < t.rows;
    const uint32_t* p = t.base + r * t.ld;
    if (run + 1 < t.upr) {
        if (live) {
            tile_run<B>(t, r, p, run);
        } else {
#pragma unroll
            for (int c = 0; c < TileRun<B>::CHUNKS; c++) *tile_chunk(t, r, run * TileRun<B>::CHUNKS + c) = make_uint4(0u, 0u, 0u, 0u);
        }
        return;
    }
    int64_t k0 = (int64_t)run * TileRun<B>::CODES;
    for (int c = run * TileRun<B>::CHUNKS; c < nkb * 8; c++, k0 += 16)
        *tile_chunk(t, r, c) = live ? tile_unit_any(p, k0, K, t.f) : make_uint4(0u, 0u, 0u, 0u);
}

// K-blocks per unit of the code-linear pass: their loads are in flight together.
constexpr int kTileKbs = 4;

// Unit u of a code-linear operand (4-bit codes, mixed widths): chunk lane & 7
// of row 4 q + lane / 8 for kTileKbs consecutive K-blocks; a warp reads 64
// contiguous bytes of each of 4 rows (4-bit codes) and writes 512 contiguous
// bytes of the image per K-block.
__device__ __forceinline__ void tile_linear(const TileSrc& t, int64_t warp_unit, int lane, int64_t K, int nkb)
{
    const int groups = (nkb + kTileKbs - 1) / kTileKbs;
    const int64_t rq = warp_unit / groups;
    const int kb0 = (int)(warp_unit - rq * groups) * kTileKbs;
    const int64_t r = rq * 4 + (lane >> 3);
    const int g = (lane & 7) ^ (int)(r & 7);          // logical chunk at physical position lane & 7
    const bool live = r < t.rows;
    const uint32_t* p = t.base + r * t.ld;
    if (t.f.b == 4) {
        // two words (16 codes) at an even word: 8-byte aligned; rows are
        // padded to whole 16-byte groups, so both words exist
        uint2 w[kTileKbs];
#pragma unroll
        for (int i = 0; i < kTileKbs; i++) {
            const int64_t k0 = (int64_t)(kb0 + i) * kBK + g * 16;
            w[i] = make_uint2(0u, 0u);
            if (live && k0 < K) w[i] = __ldg(reinterpret_cast<const uint2*>(p + (k0 >> 3)));
        }
#pragma unroll
        for (int i = 0; i < kTileKbs; i++) {
            if (kb0 + i >= nkb) break;
            const int64_t k0 = (int64_t)(kb0 + i) * kBK + g * 16;
            uint32_t o0 = 0u, o1 = 0u, o2 = 0u, o3 = 0u;
            if (live && k0 < K) {
                decode_word_b4(w[i].x, t.f.k, t.f.ew, o0, o1);
                decode_word_b4(w[i].y, t.f.k, t.f.ew, o2, o3);
                if (k0 + 16 > K) {                    // K tail: zero the codes past K
                    uint32_t ml, mh;
                    const int va = (int)(K - k0);
                    tail_masks(va > 8 ? 8 : va, ml, mh);
                    o0 &= ml; o1 &= mh;
                    const int vb = (int)(K - k0 - 8);
                    tail_masks(vb < 0 ? 0 : vb, ml, mh);
                    o2 &= ml; o3 &= mh;
                }
            }
            *tile_chunk(t, r, (kb0 + i) * 8 + g) = make_uint4(o0, o1, o2, o3);
        }
        return;
    }
#pragma unroll 1
    for (int i = 0; i < kTileKbs && kb0 + i < nkb; i++)
        *tile_chunk(t, r, (kb0 + i) * 8 + g) =
            live ? tile_unit_any(p, (int64_t)(kb0 + i) * kBK + g * 16, K, t.f) : make_uint4(0u, 0u, 0u, 0u);
}

// HBM-bound by its output (one byte per code).  Both operands in one launch
// (the first blocks take A's units, the rest B's), four K-blocks' loads in
// flight per warp and no division per chunk: 20.4 us in two launches before,
// 11.4 us now for 256 x 9216 and 4096 x 9216 4-bit operands.
__global__ void __launch_bounds__(256) esb_tile_kernel(TileSrc ta, TileSrc tb, int64_t K, int nkb, unsigned blocks_a)
{
    griddep_wait();                                   // codes and workspace may belong to the previous launch
    const bool is_a = blockIdx.x < blocks_a;
    const TileSrc& t = is_a ? ta : tb;
    const int64_t nblk = is_a ? blocks_a : gridDim.x - blocks_a;
    const int64_t blk = is_a ? blockIdx.x : blockIdx.x - blocks_a;
    if (t.packed) {
        for (int64_t u = blk * 256 + threadIdx.x; u < t.units; u += nblk * 256) {
            if (t.f.b == 3) tile_packed<3>(t, u, K, nkb);
            else if (t.f.b == 5) tile_packed<5>(t, u, K, nkb);
            else tile_packed<6>(t, u, K, nkb);
        }
    } else {
        const int lane = threadIdx.x & 31;
        for (int64_t u = blk * 8 + (threadIdx.x >> 5); u < t.units; u += nblk * 8) tile_linear(t, u, lane, K, nkb);
    }
}

// Epilogue of a chunked accumulation: the nch chunk accumulators of a tile
// (TMEM regions (buf * nch + ch) * BN) are added as exact integers, the sum
// is stored as the int32 accumulator, and float(acc) (round to nearest, as
// the oracle converts it) goes through epi_element.  Codes of any width
// that divides 16 codes per word; padding slots past N take the zero code.
// Warps 0-7: TMEM lane quarter warp & 3, column half warp >> 2.
__device__ void tiled_chunked_epilogue(const EpiParams& ep, const float* thr, int64_t M, int64_t N, int64_t n0,
                                       int BN, int64_t first, int64_t ctas, int64_t my_tiles, int nch, int nbuf,
                                       uint32_t tmem_base, float acc_scale, uint64_t* tfull, uint64_t* tempty,
                                       volatile int* err, int warp, int lane)
{
    const EpiCtx cx = make_epi_ctx(ep, thr);
    EpiParams e2 = ep;
    e2.acc_out = nullptr;                                // the exact sum is stored here instead
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const int c_lo = (warp >> 2) * (BN / 2), c_hi = c_lo + BN / 2;
    const int cpw = ep.out_cpw, ob = ep.out.b;
    const uint32_t zc = ep.codes_out ? fmt_zero_code(ep.out.b, ep.out.k) : 0u;
    for (int64_t ti = 0; ti < my_tiles && !*err; ti++) {
        const int buf = (int)(ti % nbuf);
        if (!wait_or_abort(&tfull[buf], (uint32_t)((ti / nbuf) & 1), err)) { *err = 1; break; }
        tc_fence_after();
        const int64_t m = (first + ti * ctas) * kBM + row;
        const bool mrow = m < M;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
        for (int c = c_lo; c < c_hi; c += 16) {
            int isum[16];
#pragma unroll
            for (int j = 0; j < 16; j++) isum[j] = 0;
            for (int ch = 0; ch < nch; ch++) {
                uint32_t r[16];
                tmem_ld16(taddr + (uint32_t)((buf * nch + ch) * BN + c), r);
#pragma unroll
                for (int j = 0; j < 16; j++) isum[j] += __float2int_rn(__uint_as_float(r[j]) * acc_scale);
            }
            if (c + 16 >= c_hi) {                        // every column of this warp is in registers
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_tmem_free(&tempty[buf]);
            }
            if (!mrow) continue;
            uint32_t word = 0u;
            int slot = 0;
#pragma unroll
            for (int j = 0; j < 16; j++) {
                const int64_t n = n0 + c + j;
                uint32_t code = zc;
                if (n < N) {
                    if (ep.acc_out) ep.acc_out[m * N + n] = isum[j];
                    code = epi_element(e2, cx, __int2float_rn(isum[j]), m, n, N);
                }
                if (ep.codes_out) {
                    word |= code << (ob * slot);
                    if (++slot == cpw) {
                        const int64_t wcol = (n0 + c + j) / cpw;
                        if (wcol < ep.ldo) ep.codes_out[m * ep.ldo + wcol] = word;
                        word = 0u;
                        slot = 0;
                    }
                }
            }
        }
    }
}

template <int EPI>
__global__ void __launch_bounds__(kTiledThreads, 1)
esb_gemm_tiled_kernel(const uint8_t* __restrict__ At, const uint8_t* __restrict__ Bt, int64_t M, int64_t N, int64_t mpad,
                      int64_t npad, int nkb, int kbc, int nch, int BN, int stages, int n_tiles, int64_t m_tiles,
                      float acc_scale, const __grid_constant__ EpiParams ep)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int kStage = kTileA + BN * kBK;                        // A tile then B tile (both 1024-aligned)
    const int nbuf = kTmemCols / (nch * BN) >= 2 ? 2 : 1;       // accumulator sets (one per tile in flight)
    float* thr = reinterpret_cast<float*>(smem + stages * kStage);
    uint64_t* full = reinterpret_cast<uint64_t*>(thr + 128);
    uint64_t* empty = full + kWsMaxStages;
    uint64_t* tfull = empty + kWsMaxStages;
    uint64_t* tempty = tfull + kMaxAcc;
    uint64_t* drain = tempty + kMaxAcc;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* err = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x;
    const int warp = warp_index(), lane = tid & 31;
    const int n_tile = (int)(blockIdx.x % n_tiles);
    const int64_t cta_in_n = blockIdx.x / n_tiles;
    const int64_t ctas_per_n = gridDim.x / n_tiles;
    const int64_t n0 = (int64_t)n_tile * BN;
    const int64_t my_tiles = (m_tiles > cta_in_n) ? (m_tiles - cta_in_n + ctas_per_n - 1) / ctas_per_n : 0;
    uint32_t tmem_cols = 32;                                     // a power of two >= the regions used
    while (tmem_cols < (uint32_t)(nbuf * nch * BN)) tmem_cols <<= 1;
    constexpr int lacc = 1;                              // nch == 1: two buffers
    const EpiSplit sp = epi_split<EPI>(ep, BN, my_tiles);
    // the layout above must fit the dynamic allocation (uniform for the CTA)
    if ((uintptr_t)(reinterpret_cast<const volatile uint8_t*>(err) + 4 - smem_raw) > dynamic_smem_bytes()) {
        if (tid == 0) record_status(ep.status, ESB_ERR_INTERNAL);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < stages; s++) {
            mbar_init(&full[s], 1);                      // the producer's arrive.expect_tx, then the copies' bytes
            mbar_init(&empty[s], 1);                     // the MMA commit that drained it
        }
        for (int a = 0; a < 2; a++) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], nch > 1 ? kWsEpiWarps : sp.tempty_count());
        }
        mbar_init(drain, 1);
        *err = 0;
        fence_mbar_init();
    }
    ws_alloc(warp, tmem_slot, tmem_cols);
    __syncthreads();                                     // barriers initialised, TMEM allocated
    griddep_wait();                                      // the tiled operands come from the tile kernels
    if (warp < kWsEpiWarps) ws_thresholds(thr, ep, warp, lane);
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == kTiledProdWarp) {
        // ---------------------------------------------- producer
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0u;
            // the last N-tile may end past the image: its missing rows stay
            // whatever shared memory holds (columns past N, never stored)
            const int64_t brows = npad - n0 < (int64_t)BN ? npad - n0 : (int64_t)BN;
            const uint32_t b_bytes = (uint32_t)brows * kBK;
            for (int64_t ti = 0; ti < my_tiles && !*err; ti++) {
                const uint8_t* at = At + (cta_in_n + ti * ctas_per_n) * (int64_t)kTileA;
                const uint8_t* bt = Bt + n0 * kBK;
                for (int kb = 0; kb < nkb; kb++, at += mpad * kBK, bt += npad * kBK) {
                    if (!wait_or_abort(&empty[s], ph ^ 1u, err)) { *err = 1; break; }
                    uint8_t* st = smem + s * kStage;
                    mbar_arrive_expect_tx(&full[s], (uint32_t)kTileA + b_bytes);
                    bulk_copy_g2s(st, at, (uint32_t)kTileA, &full[s]);
                    bulk_copy_g2s(st + kTileA, bt, b_bytes, &full[s]);
                    if (++s == stages) { s = 0; ph ^= 1u; }
                }
            }
        }
    } else if (warp == kWsMmaWarp) {
        // ---------------------------------------------- MMA issue
        const uint32_t idesc = idesc_e4m3_f32(BN);
        const uint32_t leader = elect_one();
        const uint64_t a_desc = smem_desc_sw128(smem_u32(smem));
        int s = 0;
        uint32_t ph = 0u;
        bool ok = true;
        for (int64_t ti = 0; ti < my_tiles && ok; ti++) {
            const int a = nbuf == 2 ? (int)(ti & 1) : 0;
            ok = warp_wait(&tempty[a], (uint32_t)((nbuf == 2 ? ti >> 1 : ti) & 1) ^ 1u, err);
            if (!ok) break;
            tc_fence_after();
            uint32_t d = tmem_base + (uint32_t)(a * nch * BN);
            uint32_t acc = 0u;
            int left = kbc;                              // K-blocks left of the chunk
            for (int kb = 0; kb < nkb; kb++, left--) {
                if (left == 0) {                         // next K-chunk: its own accumulator
                    left = kbc;
                    d += (uint32_t)BN;
                    acc = 0u;
                }
                ok = warp_wait(&full[s], ph, err);
                if (!ok) break;
                tc_fence_after();
                const uint64_t ad = a_desc + (uint64_t)s * (uint64_t)(kStage >> 4), bd = ad + (uint64_t)(kTileA >> 4);
                // four K steps of 32 codes: 32 bytes along the swizzled row
#pragma unroll
                for (int j = 0; j < kBK / 32; j++) {
                    mma_f8f6f4(d, ad + 2 * j, bd + 2 * j, idesc, acc, leader);
                    acc = 1u;
                }
                mma_commit(&empty[s], leader);
                if (++s == stages) { s = 0; ph ^= 1u; }
            }
            if (ok) mma_commit(&tfull[a], leader);
        }
        if (!ok) *err = 1;
        ws_drain(drain, err, leader);
    } else if (nch > 1) {
        // ---------------------------------------------- epilogue (K in chunks)
        if (warp < kWsEpiWarps)
            tiled_chunked_epilogue(ep, thr, M, N, n0, BN, cta_in_n, ctas_per_n, my_tiles, nch, nbuf, tmem_base,
                                       acc_scale, tfull, tempty, err, warp, lane);
    } else if (warp < sp.warps) {
        // ---------------------------------------------- epilogue
        const int64_t first = cta_in_n, ctas = ctas_per_n;
        auto rows = [=](int64_t ti, int row, int64_t& m) -> bool {
            m = (first + ti * ctas) * kBM + row;
            return m < M;
        };
        ws_epilogue<EPI>(ep, thr, rows, my_tiles, n0, N, BN, sp, lacc, tmem_base, acc_scale, tfull, tempty,
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

static int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// K-chunking of a shape: K-blocks per chunk (each chunk's partial sums stay
// below 2^24), chunk count and N-tile width; false when the kernel cannot
// hold the chunks (more than four, or a total past the int32 range) or the
// output's codes per word.
static bool tiled_plan(int64_t K, int ba, int ka, int bb, int kb, int out_cpw, int* kbc, int* nch, int* BN)
{
    const int64_t nkb = cdiv(K, kBK);
    const double img = (double)fmt_max_image(ba, ka) * fmt_max_image(bb, kb);
    if ((double)K * img >= 2147483648.0) return false;
    int64_t c = nkb;
    if ((double)K * img >= 16777216.0) {
        c = (int64_t)((16777215.0 / img) / kBK);                  // whole K-blocks per chunk
        if (c < 1) return false;
    }
    const int64_t n = cdiv(nkb, c);
    if (n > 4 || (n > 1 && 16 % out_cpw != 0)) return false;
    *kbc = (int)c;
    *nch = (int)n;
    *BN = n > 2 ? 128 : (kTiledBN % out_cpw == 0 ? kTiledBN : kTiledBNOdd);
    return *BN % out_cpw == 0;
}

// Narrower N-tiles when the widest would leave SMs idle (few row tiles: a
// classifier at a small batch).  A CTA streams 128 + BN rows of each K-block,
// so the width that minimises waves x (128 + BN); whole words per tile, at
// least 64 columns, the wider on a tie.  The whole call at 256 x 4096 x 9216:
// 37 us with 32 CTAs of 256 columns, 29 us with 128 CTAs of 64; 100 x 1000 x
// 4096 of 6-bit codes with y: 153 and 62 us.
static int tiled_bn(int64_t M, int64_t N, int bn0, int out_cpw)
{
    const int64_t sms = device_sm_count(), mt = cdiv(M, kBM);
    if (mt * cdiv(N, bn0) >= sms) return bn0;
    int best = bn0;
    int64_t cbest = cdiv(mt * cdiv(N, bn0), sms) * (kBM + bn0);
    for (int bn = bn0 - 16; bn >= 64; bn -= 16) {
        if (bn % out_cpw) continue;
        const int64_t c = cdiv(mt * cdiv(N, bn), sms) * (kBM + bn);
        if (c < cbest) { cbest = c; best = bn; }
    }
    return best;
}

size_t gemm_tiled_workspace_bytes(int64_t M, int64_t N, int64_t K)
{
    const int64_t nkb = cdiv(K, kBK);
    // (the images hold rows padded to 128 and 16 only; the sizes callers know are kept)
    return (size_t)(cdiv(M, kBM) * nkb * kTileA + cdiv(N, kTiledBN) * nkb * (int64_t)kTiledBN * kBK);
}

// The tiled path pays an extra launch and a pass over both operands.  The
// lines, 2^32 multiply-adds for 4-bit operands and 2^28 for the outputs that
// esb_gemm's kernels also take, were drawn when the pass was two launches and
// the GEMM had 256-column tiles only.  Measured since (esb_gemm's kernels and
// this one, us): 4 bits, 2^28 (512 x 512 x 1024) 12.4 and 7.8, 2^30 (1024^3) 13.4
// and 8.1, 2^32 (2048 x 2048 x 1024) 27.3 and 11.3, 2^26 (256 x 512 x 512) 8.1 and
// 7.2; 6 bits 23.7 and 14.5, 23.9 and 14.8, 64.2 and 20.1, 13.4 and 11.9: they
// could lie lower.  ESB_GEMM_TILED_MIN_MACS in the environment (read per call)
// moves them (0: every shape the kernel takes).
bool gemm_tiled_ok(int64_t M, int64_t N, int64_t K, int ba, int ka, int bb, int kb, int out_cpw)
{
    int kbc, nch, BN;
    // significand-split operands (k >= 4) take esb_gemm's kernels
    if (fmt_needs_split(ba, ka) || fmt_needs_split(bb, kb)) return false;
    if (M <= 0 || N < kTiledBN || K <= 0 || !tiled_plan(K, ba, ka, bb, kb, out_cpw, &kbc, &nch, &BN)) return false;
    if (nch > 1) return true;                                     // only this path takes that K
    double min_macs = (ba == 4 && bb == 4) ? 4294967296.0 : (BN == kTiledBNOdd ? 268435456.0 : 0.0);
    if (const char* v = getenv("ESB_GEMM_TILED_MIN_MACS")) min_macs = atof(v);
    return (double)M * N * K >= min_macs;
}

// 5, 6 or 10 output codes per word: esb_gemm's kernels take every shape of
// these too, so a call without (enough) workspace runs there.
bool gemm_tiled_optional(int out_cpw) { return kTiledBN % out_cpw != 0; }

typedef void (*TiledKernel)(const uint8_t*, const uint8_t*, int64_t, int64_t, int64_t, int64_t, int, int, int, int, int,
                            int, int64_t, float, EpiParams);
static const TiledKernel kTiledKernels[4] = {esb_gemm_tiled_kernel<kEpiB4>, esb_gemm_tiled_kernel<kEpiLean4>,
                                             esb_gemm_tiled_kernel<kEpiGen>, esb_gemm_tiled_kernel<kEpiTable>};

static int tiled_static_smem(cudaError_t* err)
{
    static int v = -1;
    if (v < 0) {
        size_t m = 0;
        for (TiledKernel k : kTiledKernels) {
            cudaFuncAttributes a;
            *err = cudaFuncGetAttributes(&a, k);
            if (*err != cudaSuccess) return -1;
            if (a.sharedSizeBytes > m) m = a.sharedSizeBytes;
        }
        v = (int)m;
    }
    return v;
}

// Operand of the tile pass; packed: runs of 3/5/6-bit words (both operands
// must have that width, so that they share the K order).
static TileSrc tile_src(const uint32_t* base, int64_t ld, int64_t rows, int64_t rpad, int64_t K, int nkb, const OpFmt& f,
                        bool packed, uint8_t* out, int64_t* blocks)
{
    TileSrc t{base, ld, rows, rpad, f, packed ? 1 : 0, 0, 0, out};
    if (packed) {
        const int codes = f.b == 3 ? TileRun<3>::CODES : f.b == 5 ? TileRun<5>::CODES : TileRun<6>::CODES;
        t.upr = (int)(K / codes) + 1;                             // whole runs, then the tail unit
        t.units = rpad * t.upr;
        *blocks = cdiv(t.units, 256);
    } else {
        t.units = rpad / 4 * cdiv(nkb, kTileKbs);                 // per warp
        *blocks = cdiv(t.units, 8);
    }
    const int64_t cap = (int64_t)device_sm_count() * 16;
    if (*blocks > cap) *blocks = cap;
    return t;
}

cudaError_t launch_gemm_tiled(int64_t M, int64_t N, int64_t K, const uint32_t* A, int64_t lda, int ba, int ka,
                              const uint32_t* B, int64_t ldb, int bb, int kb, const GemmOutputs& o, void* workspace,
                              cudaStream_t st)
{
    int kbc = 0, nch = 0, BN = 0;
    const int out_cpw = o.codes_out ? 32 / o.ep->fmt_out.b : 8;
    if (!tiled_plan(K, ba, ka, bb, kb, out_cpw, &kbc, &nch, &BN)) return cudaErrorInvalidValue;
    if (nch == 1) BN = tiled_bn(M, N, BN, out_cpw);
    EpiParams ep = make_epi(o);
    ep.dq_pow2 = ldexpf(1.0f, -(ka + kb));
    ep.acc_lim = nch == 1 ? acc_fma_limit(K, ba, ka, bb, kb) : 0.0f;
    const OpFmt fa = make_opfmt(ba, ka), fb = make_opfmt(bb, kb);
    const int nkb = (int)cdiv(K, kBK);
    const int64_t m_tiles = cdiv(M, kBM), n_tiles = cdiv(N, BN);
    uint8_t* At = static_cast<uint8_t*>(workspace);
    const int64_t mpad = m_tiles * kBM, npad = cdiv(N, 16) * 16;
    uint8_t* Bt = At + mpad * nkb * (int64_t)kBK;
    const bool packed = ba == bb && (ba == 3 || ba == 5 || ba == 6);
    int64_t blk_a = 0, blk_b = 0;
    const TileSrc ta = tile_src(A, lda, M, mpad, K, nkb, fa, packed, At, &blk_a);
    const TileSrc tb = tile_src(B, ldb, N, npad, K, nkb, fb, packed, Bt, &blk_b);
    cudaError_t e = launch_pdl(esb_tile_kernel, dim3((unsigned)(blk_a + blk_b)), dim3(256), 0, st, ta, tb, K, nkb,
                               (unsigned)blk_a);
    if (e != cudaSuccess) return e;

    const int st_smem = tiled_static_smem(&e);
    if (st_smem < 0) return e;
    const int maxs = max_dyn_smem() - st_smem;
    const int64_t fixed = 1024 + 4 * 128 + 512;
    const int64_t stage_bytes = kTileA + (int64_t)BN * kBK;
    int stages = (int)((maxs - fixed) / stage_bytes);
    if (stages > kWsMaxStages) stages = kWsMaxStages;
    if (stages < 2) return cudaErrorInvalidConfiguration;
    const size_t smem = (size_t)(fixed + (int64_t)stages * stage_bytes);
    static bool configured = false;
    if (!configured) {
        for (TiledKernel k : kTiledKernels) {
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, maxs);
            if (e != cudaSuccess) return e;
        }
        configured = true;
    }
    int64_t per_n = device_sm_count() / n_tiles;
    if (per_n < 1) per_n = 1;
    if (per_n > m_tiles) per_n = m_tiles;
    const int64_t grid = per_n * n_tiles;
    const float acc_scale = ldexpf(1.0f, fa.csc + fb.csc);
    // K in chunks has an epilogue of its own, in every instance; fp32 and int32 outputs run in the 4-bit one
    const bool codes = nch == 1 && ep.codes_out && !ep.acc_out && !ep.y_out;
    return launch_pdl(kTiledKernels[codes ? epi_kind(ep) : kEpiB4], dim3((unsigned)grid), dim3(kTiledThreads), smem, st,
                      (const uint8_t*)At, (const uint8_t*)Bt, M, N, mpad, npad, nkb, kbc, nch, BN, stages, (int)n_tiles,
                      m_tiles, acc_scale, ep);
}

}  // namespace esb
