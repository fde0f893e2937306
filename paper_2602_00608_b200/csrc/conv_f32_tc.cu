// Single-precision 3x3 convolutions (upsampling ones too) on the tensor cores: every fp32 operand is three bf16 numbers.
//
// x = x0 + x1 + x2, each the rest rounded to bf16: 8 + 8 + 8 significant bits are all 24 of x, and bf16 has fp32's exponents, so
// nothing of an operand is lost (of one below 2^-110 in size up to 2^-134, half of bf16's smallest step).  A product takes six
// bf16 products, which are exact; x1 w2 + x2 w1 + x2 w2 are left out: 2^-24 of it at most, as much as rounding it would cost
// (|x1| is up to 2^-8, |x2| up to 2^-17 of x's power of two).  The tensor core truncates its running sum at every step of K = 16,
// so a sum has two steps only, a tap of 32 channels, and the products of either size have their own: the largest, of 16 bits
// each, mostly add up exactly, and what is cut from the others is below 2^-31.  The warps that have made the operand read the sums
// and add them to their registers, smallest first, with rounding, while the next tap runs: two accumulators in turn.
// An infinite operand, or one that rounds to infinity in bf16, has parts that are NaN, and so are the sums that it is in: those are
// made anew from the operands themselves, one by one (redo_sums).  (Of the decode named below 830 -> 835 us, for the registers around
// the call; with parts that hold no NaN and a look at every sum 897, with a look where an operand asks for it 846.)
// Relative 2-norm error against 64 bits, FMA kernel (conv_f32.cu) / this one, normally distributed operands: 512->512 at 16x16 3.1e-7 /
// 1.2e-7, at 24x24 4.2e-7 / 1.7e-7, 256->256 at 48x48 4.3e-7 / 1.3e-7, 128->128 at 64x64 3.1e-7 / 1.1e-7, 32->32 at 128x128 2.3e-7 / 0.9e-7;
// sizes that spread over 2^24: 512->512 at 24x24 4.1e-7 / 1.7e-7; positive ones, whose truncations add up: 1.3e-7 / 1.0e-7 there, 0.57e-7 /
// 0.62e-7 at 8x8 (with a row of taps per sum, which is 7 % faster in the full-width 64x64 decode, 1.14e-7); one product per output 2.5e-8 / 2.6e-8.
//
// The shape is that of conv_split.cu: a cluster of S CTAs shares one tile of 16 x 8 pixels x 32 output channels, each takes 1/S of
// the 32-channel chunks, the partial sums meet in distributed shared memory, statistics are records.  A chunk's operand is
// three tiles of 180 halo pixels x 32 channels (64-byte rows, swizzled), written once and read by nine taps through views; a
// tap's weights are one box of 96 rows, the parts one above the other, so that x0 takes one MMA of N = 96 with all three, x1 one
// of 64 and x2 one of 32, each added where products of that size are.  Two CTAs share an SM.  Bound by the taps' hand-over (issue,
// sum, barrier) and by the chain of latencies around it.
// us, launches of a decode, FMA kernel -> this one: 512->512 at 8x8 28.9 -> 26.8, at 16x16 43.4 -> 29.0, upsampling to 16x16 30.6 -> 27.5, to
// 32x32 76.0 -> 45.0; 512->256 at 32x32 76.1 -> 45.4, 256->256 43.2 -> 29.0, 128->128 at 64x64 45.4 -> 31.0; 32->32 on four 256x256
// frames 142 -> 113, at 128x128 45 -> 37.  Decodes: 64x64 of the full-width layout 1252 -> 835 us, sixteen 256x256 frames of the small
// one 2765 -> 2216.
#include <string.h>

#include <algorithm>

#include "conv_cluster.cuh"
#include "conv_tile.cuh"
#include "tc_pair.cuh"

namespace vd {

namespace {

using namespace cc;
using namespace tc;
using convtile::NPIX;
using convtile::PW;
using convtile::TILE_H;
using convtile::TILE_W;

constexpr int kWarps = 10, kThreads = kWarps * 32;           // MMA, weights, eight producer / epilogue warps
constexpr int kProd0 = 2, kProd = 8 * 32;
constexpr int BN = 32, kChunk = 32, ROWS = TILE_H * TILE_W;  // output channels of a cluster, input channels of a chunk, rows of a tile
constexpr int kMaxB = 9, kMaxSlice = 512;                    // weight stages; input channels of a CTA
constexpr int PARTS = 3;                                     // bf16 numbers of an operand
constexpr int ROW_BYTES = kChunk * 2;                        // a pixel's, or an output channel's, part: 64 bytes (64-byte swizzle)
constexpr int A_PART_BYTES = (NPIX * ROW_BYTES + 1023) / 1024 * 1024, A_BYTES = PARTS * A_PART_BYTES, B_BYTES = PARTS * BN * ROW_BYTES;
constexpr int ACCS = 2, ACC_COLS = 128;                      // accumulators of a tap each, in turn: columns [x0 w0 | x0 w1 + x1 w0 | x0 w2 + x1 w1 + x2 w0]
constexpr int kTailBytes = 2 * kMaxSlice * 4 + 320;

enum { K3X3 = 0, KPHASE = 1 };
__host__ __device__ constexpr int taps_of(int kind) { return kind == K3X3 ? 9 : 4; }

struct TBars {
    uint64_t a_full, a_empty;
    uint64_t b_full[kMaxB], b_empty[kMaxB];
    uint64_t t_full[ACCS], t_empty[ACCS];
    uint64_t acc_full, rx_full;
    uint32_t tmem_base, abort_flag, unused;
};
static_assert(sizeof(TBars) <= 320, "barrier block");
struct TShape { int splits, n_b, tail_off; };

// the next parts of two numbers (the first in the low half), the largest first; the rests stay
__device__ __forceinline__ uint32_t take_bf16(float& v0, float& v1) {
    const uint32_t p = pack_bf16(v0, v1);
    v0 -= __uint_as_float(p << 16);
    v1 -= __uint_as_float(p & 0xffff0000u);
    return p;
}
// 16-byte piece c of row R of a partial: eight rows of a piece, and four rows of two pieces side by side, are on distinct banks
__device__ __forceinline__ int exchange_piece(int R, int c) { return c ^ ((R & 3) * 2 + ((R >> 2) & 1)); }
__device__ __forceinline__ void commit_to_cluster(uint32_t bar, uint16_t mask, uint32_t on) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n"
                 ::"r"(bar), "h"(mask), "r"(on) : "memory");
}

// The operand of one tile, made by eight warps: 18x10 halo pixels x 32 channels a chunk, an entry is (pixel, 4 channels).
struct Operand {
    static constexpr int N = (NPIX * 8 + kProd - 1) / kProd;
    int goff[N];                                             // element offset of the entry's source pixel
    uint32_t soff, vm;                                       // where entry 0 goes (entry e: e * kProd * 8 on); entries inside the image
    const float* xb;
    float4 raw[N];
    __device__ __forceinline__ void prepare(const ConvArgs& a, int frame, int c_first, int ty, int tx, int H, int W, int ptid) {
        const int j = ptid & 7, pix0 = ptid >> 3;
        soff = (uint32_t)(pix0 * ROW_BYTES + (((j >> 1) ^ (pix0 >> 1 & 3)) << 4) + (j & 1) * 8);
        vm = 0u;
#pragma unroll
        for (int e = 0; e < N; ++e) {
            const int pix = (e * kProd + ptid) >> 3, py = pix / PW, px = pix - py * PW;
            const int oy = ty + py - 1, ox = tx + px - 1;
            const bool v = oy >= 0 && oy < H && ox >= 0 && ox < W && pix < NPIX;
            vm |= (v ? 1u : 0u) << e;
            goff[e] = v ? (oy * W + ox) * a.Cin : 0;
        }
        xb = (const float*)a.x + (size_t)frame * H * W * a.Cin + c_first + j * 4;
    }
    __device__ __forceinline__ void load(int u) {
#pragma unroll
        for (int e = 0; e < N; ++e)
            if (vm >> e & 1u) raw[e] = __ldcg((const float4*)(xb + (size_t)u * kChunk + goff[e]));
    }
    __device__ __forceinline__ void transform(uint8_t* dst, int u, bool prologue, bool silu, const float* s_scale, const float* s_shift, int ptid) {
        float4 sc = make_float4(1.f, 1.f, 1.f, 1.f), sf = make_float4(0.f, 0.f, 0.f, 0.f);
        if (prologue) {
            const int c = u * kChunk + (ptid & 7) * 4;
            sc = *(const float4*)(s_scale + c);
            sf = *(const float4*)(s_shift + c);
        }
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (e == N - 1 && ((e * kProd + ptid) >> 3) >= NPIX) break;
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (vm >> e & 1u) {                              // outside the image the transformed tensor is zero
                const float x[4] = {raw[e].x, raw[e].y, raw[e].z, raw[e].w}, s4[4] = {sc.x, sc.y, sc.z, sc.w}, f4[4] = {sf.x, sf.y, sf.z, sf.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    v[q] = x[q];
                    if (prologue) v[q] = fmaf(v[q], s4[q], f4[q]);
                    if (silu) v[q] = v[q] / (1.0f + expf(-v[q]));
                }
            }
            uint8_t* d = dst + soff + e * (kProd * 8);
#pragma unroll
            for (int p = 0; p < PARTS; ++p) {
                const uint32_t lo = take_bf16(v[0], v[1]), hi = take_bf16(v[2], v[3]);
                *(uint2*)(d + p * A_PART_BYTES) = make_uint2(lo, hi);
            }
        }
    }
};

// Those of a thread's sixteen partial sums (one pixel, channels [16 h, 16 h + 16) of the CTA's block) that are NaN, in plain fp32.
// It works everything out for itself: what it would be handed would be kept in registers where they are short.
template <int KIND>
__device__ __noinline__ void redo_sums(const ConvArgs& a, const TShape& sh) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const float* s_scale = (const float*)(smem + sh.tail_off);
    const float* s_shift = s_scale + kMaxSlice;
    constexpr int TAPS = taps_of(KIND), COLS = KIND == K3X3 ? 3 : 2;
    const int S = sh.splits, rank = S > 1 ? (int)cluster_ctarank() : 0;
    const int H = KIND == KPHASE ? a.Hs : a.H, W = KIND == KPHASE ? a.Ws : a.W;
    const int tiles_x = (W + TILE_W - 1) / TILE_W, tiles = tiles_x * ((H + TILE_H - 1) / TILE_H), nblk = a.Cout / BN;
    int item = (int)blockIdx.x / S;
    const int blk = item % nblk;
    item /= nblk;
    const int par = KIND == KPHASE ? (item & 3) : 0;
    if (KIND == KPHASE) item >>= 2;
    const int tile = item % tiles, frame = item / tiles;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31, R = (warp & 3) * 32 + lane, h = (warp - kProd0) >> 2;
    float* row = (float*)smem + R * BN;
    const int y = (tile / tiles_x) * TILE_H + (R >> 3), x = (tile % tiles_x) * TILE_W + (R & 7);
    if (y >= H || x >= W) return;
    const int kchunks = a.Cin / kChunk, k0 = rank * kchunks / S, nch = ((rank + 1) * kchunks / S - k0) * kChunk;
    const float* image = (const float*)a.x + (size_t)frame * H * W * a.Cin + k0 * kChunk;
    const bool prologue = a.scale != nullptr || a.in_rec != nullptr;
    // A NaN among the operands ends it: a frame of them costs one product per sum, beginning with the tap that reads the pixel itself.
    const int centre = KIND == KPHASE ? (par ^ 3) : 4;
#pragma unroll 1
    for (int o = 0; o < 16; ++o) {
        float* at = row + exchange_piece(lane, h * 4 + (o >> 2)) * 4 + (o & 3);
        if (!isnan(*at)) continue;
        float sum = 0.f;
#pragma unroll 1
        for (int t = 0; t < TAPS && !isnan(sum); ++t) {
            const int tap = (t + centre) % TAPS;
            const int sy = y - 1 + (KIND == KPHASE ? par >> 1 : 0) + tap / COLS, sx = x - 1 + (KIND == KPHASE ? par & 1 : 0) + tap % COLS;
            const bool inside = sy >= 0 && sy < H && sx >= 0 && sx < W;
            const __nv_bfloat16* w = (const __nv_bfloat16*)a.w + (((size_t)(par * TAPS + tap) * nblk + blk) * (PARTS * BN) + h * 16 + o) * a.Cin + k0 * kChunk;
#pragma unroll 1
            for (int c = 0; c < nch && !isnan(sum); ++c) {
                float v = 0.f, weight = 0.f;
                if (inside) {
                    v = __ldcg(image + ((size_t)sy * W + sx) * a.Cin + c);
                    if (prologue) v = fmaf(v, s_scale[c], s_shift[c]);
                    if (a.silu) v = v / (1.0f + expf(-v));
                }
                for (int p = PARTS - 1; p >= 0; --p) weight += __bfloat162float(w[(size_t)p * BN * a.Cin + c]);
                sum = fmaf(v, weight, sum);
            }
        }
        *at = sum;
    }
}

template <int KIND>
__global__ void __launch_bounds__(kThreads, 2)
conv_f32_tc_kernel(const __grid_constant__ ConvArgs a, const __grid_constant__ TShape sh, const __grid_constant__ CUtensorMap tm_w, unsigned int* status) {
    constexpr int TAPS = taps_of(KIND);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int n_b = sh.n_b, S = sh.splits;
    uint8_t* smem_a = smem;
    uint8_t* smem_b = smem + A_BYTES;
    // over the operand stages, once every MMA of the cluster is done: this CTA's partials [ROWS][BN], and those of its
    // rows [S][rows][BN]
    float* part = (float*)smem;
    float* rx = S > 1 ? part + ROWS * BN : part;
    float* s_scale = (float*)(smem + sh.tail_off);
    float* s_shift = s_scale + kMaxSlice;
    TBars* bars = (TBars*)(s_shift + kMaxSlice);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = S > 1 ? (int)cluster_ctarank() : 0;

    // ---- this cluster's item: (frame, tile, output parity, channel block); for KPHASE the tile grid is that of the source
    const int H = KIND == KPHASE ? a.Hs : a.H, W = KIND == KPHASE ? a.Ws : a.W;
    const int tiles_x = (W + TILE_W - 1) / TILE_W, tiles = tiles_x * ((H + TILE_H - 1) / TILE_H);
    const int nblk = a.Cout / BN;
    int item = (int)blockIdx.x / S;
    const int blk = item % nblk, n0 = blk * BN;
    item /= nblk;
    const int par = KIND == KPHASE ? (item & 3) : 0;
    if (KIND == KPHASE) item >>= 2;
    const int tile = item % tiles, frame = item / tiles;
    const int ty = (tile / tiles_x) * TILE_H, tx = (tile % tiles_x) * TILE_W;
    const int kchunks = a.Cin / kChunk;
    const int k0 = rank * kchunks / S, nk = (rank + 1) * kchunks / S - k0;           // chunks of this CTA
    const int loads = nk * TAPS;

    if (tid == 0) {
        mbar_init(smem_u32(&bars->a_full), 8);
        mbar_init(smem_u32(&bars->a_empty), 1);
        for (int i = 0; i < n_b; ++i) { mbar_init(smem_u32(&bars->b_full[i]), 1); mbar_init(smem_u32(&bars->b_empty[i]), 1); }
        for (int i = 0; i < ACCS; ++i) { mbar_init(smem_u32(&bars->t_full[i]), 1); mbar_init(smem_u32(&bars->t_empty[i]), 8); }
        mbar_init(smem_u32(&bars->acc_full), S);             // one commit from every CTA of the cluster
        mbar_init(smem_u32(&bars->rx_full), 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(smem_u32(&bars->rx_full), ROWS * BN * 4);  // this CTA's rows from all S partials
    }
    if (warp == 0) tmem_alloc(smem_u32(&bars->tmem_base), ACCS * ACC_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    cluster_arrive();                                        // (waited for before anything is sent to another CTA)
    griddep_launch();

    if (warp == 1) {
        // ------------------------------------------------ weights (they do not depend on the kernel before)
        if (lane == 0) {
            uint32_t st = 0, ph = 0;
            int issued = 0;
            bool ok = true;
            for (int u = 0; u < nk && ok; ++u) {
#pragma unroll 1
                for (int tap = 0; tap < TAPS; ++tap) {
                    if (issued >= n_b) ok = mbar_wait(smem_u32(&bars->b_empty[st]), ph ^ 1, abort_flag);
                    if (!ok) break;
                    const uint32_t full = smem_u32(&bars->b_full[st]);
                    mbar_arrive_expect_tx(full, B_BYTES);
                    tma_load_2d(smem_u32(smem_b + st * B_BYTES), &tm_w, (k0 + u) * kChunk, ((par * TAPS + tap) * nblk + blk) * (PARTS * BN), full);
                    ++issued;
                    if (++st == (uint32_t)n_b) { st = 0; ph ^= 1; }
                }
            }
            // what a CTA that gave up has on its way lands before the others may leave (the last arrival below)
            (void)mbar_wait(smem_u32(&bars->acc_full), 0, abort_flag);
            if (*abort_flag) land_loads(bars->b_full, n_b, issued);
        }
        __syncwarp();
        cluster_wait();
    } else if (warp == 0) {
        // ------------------------------------------------ MMA issue (warp-uniform, predicated on one elected lane)
        const uint32_t lead = elect_one();
        constexpr uint32_t idesc3 = make_idesc_bf16(128, 3 * BN), idesc2 = make_idesc_bf16(128, 2 * BN), idesc1 = make_idesc_bf16(128, BN);
        constexpr uint32_t SWIZZLE_64B = 4;
        const uint32_t a_desc = desc_hi(PW * ROW_BYTES, SWIZZLE_64B), b_desc = desc_hi(8 * ROW_BYTES, SWIZZLE_64B);
        const uint32_t a_lo0 = desc_lo(smem_u32(smem_a)), b_lo0 = desc_lo(smem_u32(smem_b));
        uint32_t bs = 0, bph = 0;
        int used = 0;                                        // (a stage that no later load needs is not handed back)
        auto wait_on = [&](uint64_t* b, uint32_t ph) {
            if (!mbar_try_wait(smem_u32(b), ph)) (void)mbar_wait(smem_u32(b), ph, abort_flag);
            tc_fence_after();
        };
#pragma unroll 1
        for (int u = 0; u < nk; ++u) {
            if (*abort_flag) break;
            wait_on(&bars->a_full, (uint32_t)u & 1u);
            constexpr uint32_t PIX = ROW_BYTES >> 4, PART = A_PART_BYTES >> 4;
            uint32_t a0 = a_lo0 + (KIND == KPHASE ? (uint32_t)((par >> 1) * PW + (par & 1)) * PIX : 0u);
            constexpr int COLS = KIND == K3X3 ? 3 : 2;
            int kx = 0;
#pragma unroll 1
            for (int tap = 0; tap < TAPS; ++tap, ++used) {
                wait_on(&bars->b_full[bs], bph);
                const uint32_t b = b_lo0 + bs * (uint32_t)(B_BYTES >> 4);
                const int acc = used & (ACCS - 1);
                const uint32_t td = tmem + (uint32_t)(acc * ACC_COLS);
                wait_on(&bars->t_empty[acc], (uint32_t)((used / ACCS) & 1) ^ 1u);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    umma_bf16_split_on(td, a0 + 2 * k, a_desc, b + 2 * k, b_desc, idesc3, k == 0 ? 0u : 1u, lead);
                    umma_bf16_split_on(td + BN, a0 + PART + 2 * k, a_desc, b + 2 * k, b_desc, idesc2, 1u, lead);
                    umma_bf16_split_on(td + 2 * BN, a0 + 2 * PART + 2 * k, a_desc, b + 2 * k, b_desc, idesc1, 1u, lead);
                }
                umma_commit_on(smem_u32(&bars->t_full[acc]), lead);
                if (used + 1 + n_b <= loads) umma_commit_on(smem_u32(&bars->b_empty[bs]), lead);
                __syncwarp();
                if (++bs == (uint32_t)n_b) { bs = 0; bph ^= 1; }
                if (++kx == COLS) { kx = 0; a0 += (uint32_t)(PW - COLS + 1) * PIX; } else a0 += PIX;
            }
            if (u + 1 < nk) umma_commit_on(smem_u32(&bars->a_empty), lead);
            __syncwarp();
        }
        __syncwarp();
        cluster_wait();
        commit_to_cluster(smem_u32(&bars->acc_full), (uint16_t)((1u << S) - 1u), lead);
        __syncwarp();
        if (*abort_flag) (void)wait_cluster(smem_u32(&bars->acc_full), 0, abort_flag);       // (the others no longer wait for the products under way)
        __syncwarp();
    } else {
        // ------------------------------------------------ operand prologue, and the taps' sums
        const int ptid = tid - kProd0 * 32, pw = warp - kProd0;
        const bool prologue = a.scale != nullptr || a.in_rec != nullptr, silu = a.silu != 0;
        const int nch = nk * kChunk;
        Operand op;
        op.prepare(a, frame, k0 * kChunk, ty, tx, H, W, ptid);
        InputStats stats;
        if (a.in_rec) stats.prepare(a, frame, k0 * kChunk, nch, pw, lane, s_scale, s_shift);
        if (pw == 0) touch_params(a, &bars->unused);
        griddep_wait();
        if (a.in_rec) stats.load(a, lane);
        op.load(0);
        const int h = pw >> 2, R0 = (warp & 3) * 32;         // the warp's share of an accumulator: 32 rows x 16 channels
        const uint32_t tacc = tmem + (uint32_t)(h * 16) + ((uint32_t)R0 << 16);
        float v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = 0.f;
        int used = 0;
        bool ok = true;
#pragma unroll 1
        for (int u = 0; u < nk && ok; ++u) {
            if (u == 0 && prologue) {
                if (a.in_rec) stats.finish(a, nch, lane, 1.f, s_scale, s_shift);
                else
                    for (int c = ptid; c < nch; c += kProd) {
                        s_scale[c] = __ldcg(a.scale + (size_t)frame * a.Cin + k0 * kChunk + c);
                        s_shift[c] = __ldcg(a.shift + (size_t)frame * a.Cin + k0 * kChunk + c);
                    }
                named_barrier_sync(1, kProd);
            }
            if (u > 0 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->a_empty), (uint32_t)(u - 1) & 1u, abort_flag))) break;
            op.transform(smem_a, u, prologue, silu, s_scale, s_shift, ptid);
            if (u + 1 < nk) op.load(u + 1);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars->a_full));
#pragma unroll 1
            for (int tap = 0; tap < TAPS; ++tap, ++used) {
                const int acc = used & (ACCS - 1);
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->t_full[acc]), (uint32_t)(used / ACCS) & 1u, abort_flag));
                if (!ok) break;
                tc_fence_after();
                const uint32_t at = tacc + (uint32_t)(acc * ACC_COLS);
                uint32_t r[16], t[16];                       // smallest terms first
                tmem_ld16(at + 2 * BN, r);
                tmem_ld16(at + BN, t);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 16; ++c) r[c] = __float_as_uint(__uint_as_float(r[c]) + __uint_as_float(t[c]));
                tmem_ld16(at, t);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars->t_empty[acc]));           // (in registers: the accumulator may go)
#pragma unroll
                for (int c = 0; c < 16; ++c) v[c] += __uint_as_float(t[c]) + __uint_as_float(r[c]);
            }
        }
        // ------------------------------------------------ exchange and epilogue: row R of the tile belongs to CTA R / rpo
        const int rpo_log2 = 7 - (__ffs(S) - 1), rpo = 1 << rpo_log2;                 // (S is a power of two)
        static_assert(ROWS == 128, "rows of a tile");
        auto exchange = [&] {
            (void)mbar_wait(smem_u32(&bars->acc_full), 0, abort_flag);       // every CTA of the cluster is done with its operands
            tc_fence_after();
            __syncwarp();
            cluster_wait();
            float* row = part + (R0 + lane) * BN;
#pragma unroll
            for (int c = 0; c < 4; ++c) *(float4*)(row + exchange_piece(lane, h * 4 + c) * 4) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
            bool odd = false;
#pragma unroll
            for (int c = 0; c < 16; ++c) odd |= isnan(v[c]);
            if (odd) redo_sums<KIND>(a, sh);
            __syncwarp();
            fence_proxy_async_smem();
            named_barrier_sync(1, kProd);
            if (S > 1) {                                     // an owner's rows lie together
                if (ptid < S)
                    copy_to_peer(map_to_cta(smem_u32(rx + rank * rpo * BN), (uint32_t)ptid), smem_u32(part + ptid * rpo * BN), (uint32_t)(rpo * BN * 4),
                                 map_to_cta(smem_u32(&bars->rx_full), (uint32_t)ptid));
                __syncwarp();
                (void)wait_cluster(smem_u32(&bars->rx_full), 0, abort_flag);
            }
            __syncwarp();
            cluster_arrive();                                // what is sent to this CTA has landed
        };
        finish_rows<BN, 2>(a, [&](int s, int local, int c) { return rx + (s * rpo + local) * BN + exchange_piece(rank * rpo + local, c) * 4; }, S, rpo, ptid, frame, n0,
                           KIND == KPHASE ? 2 * H : H, KIND == KPHASE ? 2 * W : W, (KIND == KPHASE ? tile * 4 + par : tile) * S + rank,
                           [&](int local, int& oy, int& ox) -> bool {
                               const int R = rank * rpo + local;
                               oy = ty + (R >> 3);
                               ox = tx + (R & 7);
                               const bool valid = oy < H && ox < W;
                               if (KIND == KPHASE) { oy = 2 * oy + (par >> 1); ox = 2 * ox + (par & 1); }
                               return valid;
                           },
                           exchange);
    }
    __syncwarp();
    if (warp < kProd0) cluster_arrive();
    cluster_wait();                                          // the sources of this CTA's copies may go; its accumulators have been read
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, ACCS * ACC_COLS);
    }
    if (tid == kProd0 * 32 && bars->abort_flag && status) {
        if (atomicCAS(status, 0u, kStatusConvTimeout) == 0u) {
            status[1] = blockIdx.x;
            status[2] = (uint32_t)BN;
        }
    }
}

// OIHW -> bf16 [tap][block of 32 output channels][part][32][Cin]; phase: the sixteen taps of the phase-collapsed upsampling form
// (parity * 4 + dy * 2 + dx, each the sum of the 3x3 taps that read the same source pixel, in conv_f32.cu's order).
template <typename T>
__global__ void pack_weight_f32_tc_kernel(const T* w, __nv_bfloat16* packed, int Cout, int Cin, int taps, bool phase) {
    const int64_t total = (int64_t)taps * Cout * Cin;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % Cin), o = (int)((i / Cin) % Cout), tap = (int)(i / ((int64_t)Cin * Cout));
        int ky0 = tap / 3, ky1 = ky0, kx0 = tap % 3, kx1 = kx0;
        if (phase) {
            const int pa = tap >> 3, pb = (tap >> 2) & 1, dy = (tap >> 1) & 1, dx = tap & 1;
            ky0 = dy == 0 ? 0 : 1 + pa; ky1 = dy == 0 ? pa : 2; kx0 = dx == 0 ? 0 : 1 + pb; kx1 = dx == 0 ? pb : 2;
        }
        float v = 0.f;
        for (int ky = ky0; ky <= ky1; ++ky)
            for (int kx = kx0; kx <= kx1; ++kx) {
                const size_t j = ((size_t)o * Cin + c) * 9 + ky * 3 + kx;
                v += sizeof(T) == 2 ? __bfloat162float(((const __nv_bfloat16*)w)[j]) : ((const float*)w)[j];
            }
        const size_t row = ((size_t)tap * (Cout / BN) + o / BN) * (PARTS * BN) + o % BN;
        for (int p = 0; p < PARTS; ++p) {
            // (the parts add up to the weight: an infinity is its first part, and what would round up to one is cut)
            const bool cut = fabsf(v) >= 3.39617752e38f;     // 2^128 (1 - 2^-9)
            const __nv_bfloat16 part = cut ? __ushort_as_bfloat16((unsigned short)(__float_as_uint(v) >> 16)) : __float2bfloat16_rn(v);
            packed[(row + p * BN) * Cin + c] = part;
            v = isinf(v) ? 0.f : v - __bfloat162float(part);
        }
    }
}

int kind_of(const ConvArgs& a) { return a.upsample == 2 ? KPHASE : K3X3; }
int tiles_of(const ConvArgs& a) {
    const int h = a.upsample == 2 ? a.Hs : a.H, w = a.upsample == 2 ? a.Ws : a.W;
    return ((w + TILE_W - 1) / TILE_W) * ((h + TILE_H - 1) / TILE_H);
}

template <int KIND> struct Build {
    static cudaError_t launch(const ConvArgs& a, const ConvF32TcPlan& p, unsigned int* status, cudaStream_t s) {
        const long long ctas = (long long)tiles_of(a) * (a.Cout / BN) * (KIND == KPHASE ? 4 : 1) * a.B * p.splits;
        return launch_clusters<conv_f32_tc_kernel<KIND>>({ctas, kThreads, p.smem, kSplitSmemMax, p.splits}, s, a, TShape{p.splits, p.n_b, p.tail_off},
                                                         *(const CUtensorMap*)p.tmap, status);
    }
    static bool fits(const ConvF32TcPlan& p) { return clusters_fit<conv_f32_tc_kernel<KIND>>(kThreads, kSplitSmemMax, p.splits); }
};
template <class F> auto with_build(const ConvArgs& a, F f) { return kind_of(a) == K3X3 ? f(Build<K3X3>()) : f(Build<KPHASE>()); }

}  // namespace

bool conv_f32_tc_supported(const ConvArgs& a) {
    if (!conv_f32_supported(a) || a.bf16_operands || a.ksize != 3 || a.Cin % kChunk != 0 || a.Cout % BN != 0) return false;
    return (long long)a.Hs * a.Ws * a.Cin <= 0x7fffffffLL;   // 32-bit element offsets within a frame
}

// K divided among a cluster as long as two CTAs per SM are not exceeded.
bool conv_f32_tc_choose(const ConvArgs& a, ConvF32TcPlan* p, int max_splits) {
    p->valid = 0;
    if (!conv_f32_tc_supported(a)) return false;
    const int kind = kind_of(a), kchunks = a.Cin / kChunk;
    const long long ctas = (long long)tiles_of(a) * (a.Cout / BN) * (kind == KPHASE ? 4 : 1) * std::max(a.B, 1);
    int s = 1;
    while (s < max_splits && 2 * s <= kchunks && ctas * 2 * s <= 296) s *= 2;
    const int nk = (kchunks + s - 1) / s;
    if (nk * kChunk > kMaxSlice) return false;
    p->splits = s;
    p->n_b = std::min(std::min(nk * taps_of(kind), kMaxB), (kSplitSmemMax - 1024 - kTailBytes - A_BYTES) / B_BYTES);
    p->tail_off = (std::max(A_BYTES + p->n_b * B_BYTES, (s > 1 ? 2 : 1) * ROWS * BN * 4) + 15) / 16 * 16;
    p->smem = p->tail_off + kTailBytes + 1024;
    return p->n_b >= 1 && p->smem <= kSplitSmemMax;
}

// Narrow layers of few tiles stay on the FMA kernel: there a layer is the chain of latencies, which the taps' hand-over lengthens.
// us, FMA kernel / this one, the same layer again and again: 64 channels, 1 tile 10.3 / 12.4, 2 tiles 11.9 / 13.8, 24 16.5 / 14.4,
// 48 24.6 / 18.1, 72 24.6 / 18.5, 128 39.0 / 25.1; upsampling, tiles times parities, 32 12.4 / 12.4, 64 18.5 / 14.8, 96 26.7 / 20.5, 128 26.7 /
// 20.6; 32 channels, 24 tiles 12.4 / 14.2, 48 and 72 12.4 / 14.4, 96 16.4 / 14.4, 128 16.5 / 14.4.  From 128 on this one gains in all of them.
// 128 channels: 1 tile 10.3 / 12.4, 2 tiles 12.4 / 13.3, 32 39.0 / 25.6; 512 from the smallest on (24.7 / 22.6).
bool conv_f32_tc_pays(const ConvArgs& a) {
    return a.Cin >= 128 || (long long)tiles_of(a) * (a.upsample == 2 ? 4 : 1) * std::max(a.B, 1) >= 128;
}

bool conv_f32_tc_fits(const ConvArgs& a, const ConvF32TcPlan& p) {
    return with_build(a, [&](auto build) { return build.fits(p); });
}

int conv_f32_tc_slots(const ConvArgs& a, const ConvF32TcPlan& p, int groups) {
    return tiles_of(a) * (a.upsample == 2 ? 4 : 1) * p.splits * rec_parts(BN, a.Cout / groups);
}

size_t conv_f32_tc_packed_bytes(int Cout, int Cin, bool phase) { return (size_t)(phase ? 16 : 9) * Cout * Cin * PARTS * 2; }

cudaError_t conv_f32_tc_prepare(const ConvArgs& a, ConvF32TcPlan* p) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t d[2] = {(cuuint64_t)a.Cin, (cuuint64_t)(a.upsample == 2 ? 16 : 9) * a.Cout * PARTS};
    const cuuint64_t st[1] = {(cuuint64_t)a.Cin * 2};
    const cuuint32_t box[2] = {kChunk, PARTS * BN};
    const cuuint32_t one[2] = {1, 1};
    if (enc((CUtensorMap*)p->tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(a.w), d, st, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    p->valid = 1;
    return cudaSuccess;
}

cudaError_t launch_conv_f32_tc(const ConvArgs& a, const ConvF32TcPlan& p, unsigned int* status, cudaStream_t s) {
    if (!p.valid) return cudaErrorInvalidValue;
    if (a.in_rec && !rec_groups_ok(a.Cin, a.in_G)) return cudaErrorInvalidValue;
    if (a.out_rec && !rec_groups_ok(a.Cout, a.out_G)) return cudaErrorInvalidValue;
    return with_build(a, [&](auto build) { return build.launch(a, p, status, s); });
}

cudaError_t launch_pack_weight_f32_tc(const void* w, int w_dtype, void* packed, int Cout, int Cin, bool phase, cudaStream_t s) {
    const int t = phase ? 16 : 9;
    const int grid = (int)std::min<int64_t>(((int64_t)t * Cout * Cin + 255) / 256, 148 * 16);
    if (w_dtype == VD_BF16) pack_weight_f32_tc_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>((const __nv_bfloat16*)w, (__nv_bfloat16*)packed, Cout, Cin, t, phase);
    else pack_weight_f32_tc_kernel<float><<<grid, 256, 0, s>>>((const float*)w, (__nv_bfloat16*)packed, Cout, Cin, t, phase);
    return cudaGetLastError();
}

}  // namespace vd
