// Convolutions of small images: the implicit GEMM of conv_tc.cu divided along its K dimension.
//
// conv_tc.cu gives a CTA a 16x8-pixel tile and all of K.  A 512-channel layer of an 8x8 image is then two CTAs, each of
// which walks 8 chunks x 9 taps on its own while 146 SMs idle, and a GroupNorm pass stands between every two layers.
// Here a layer is cut into work for the whole GPU and needs no other launch:
//   * a cluster of S CTAs shares one (tile, block of 64 output channels): each takes 1/S of the 64-channel chunks, and
//     the partial accumulators meet in distributed shared memory (conv_cluster.cuh);
//   * nothing is persistent: weights do not depend on the kernel before, so a CTA streams as many of them as its
//     shared memory holds while that kernel is still running (programmatic dependent launch), and two CTAs fit
//     an SM, so the next layer's CTAs set themselves up beside this layer's;
//   * GroupNorm statistics are records of the producing layer's CTAs, merged while the first input tile is on its way.
// Such a layer is a chain of latencies (input, transform, MMAs, exchange, output), each run once, so the code is kept
// small where it can be: straight-line code that runs once costs its instruction fetches.
// Operand layouts (18x10-pixel halo tile, tap views, 128-byte swizzle), packed weights and rounding points are those of
// conv_tc.cu; only the order of the fp32 sums differs.
#include <cuda_fp16.h>
#include <string.h>

#include <algorithm>

#include "conv_cluster.cuh"
#include "conv_tile.cuh"
#include "tc_pair.cuh"

namespace vd {

namespace {

using namespace cc;
using namespace tc;
using convtile::A_TILE_BYTES;
using convtile::ITEMS;
using convtile::NPIX;
using convtile::PW;
using convtile::TILE_H;
using convtile::TILE_W;

constexpr int kWarps = 10, kThreads = kWarps * 32;           // MMA, weights, eight producer / epilogue warps
constexpr int kProd0 = 2, kProd = 8 * 32;
constexpr int kMaxA = 2, kMaxB = 10;
constexpr int kMaxSliceC = 512;                              // channels of one CTA's K slice
constexpr int kTailBytes = 2 * kMaxSliceC * 4 + 256;         // after the operand stages: scale/shift of the slice, barriers

enum { K3X3 = 0, K1X1 = 1, KPHASE = 2 };
__host__ __device__ constexpr int taps_of(int kind) { return kind == K3X3 ? 9 : (kind == K1X1 ? 1 : 4); }

struct SBars {
    uint64_t a_full[kMaxA], a_empty[kMaxA];
    uint64_t b_full[kMaxB], b_empty[kMaxB];
    uint64_t acc_full, rx_full;
    uint32_t tmem_base, abort_flag, unused;
};

// 16-byte piece c of row R of a partial lies at this piece: eight rows of a piece, and four rows of two pieces side by side,
// are on distinct banks.
template <int BN> __device__ __forceinline__ int exchange_piece(int R, int c) { return BN < 64 ? c : c ^ ((R & 3) * 2 + ((R >> 2) & 1)); }

// arrives, once the MMAs issued so far have completed, on the barrier at this offset in every CTA of `mask`
__device__ __forceinline__ void commit_to_cluster(uint32_t bar, uint16_t mask, uint32_t on) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n"
                 ::"r"(bar), "h"(mask), "r"(on) : "memory");
}

// The operand of one tile, made by NPW warps: 18x10 halo pixels x 64 channels a chunk, an entry is (pixel, 8 channels).
// fp32 input: four channels from the chunk's first half, four from its second.  `prepare` is what depends on the thread
// alone; an entry's registers take the next chunk's values as soon as they have been read (515 -> 465 us for one 64x64
// frame, most of whose layers give a CTA two chunks).
template <int KIND, bool IN_BF16, int NPW> struct Operand {
    static constexpr int NT = NPW * 32, N = (ITEMS + NT - 1) / NT, ESZ = IN_BF16 ? 2 : 4, HALVES = IN_BF16 ? 1 : 2, NV = 8 / HALVES;
    static_assert(NT / 8 % 8 == 0, "an entry's swizzle is the first one's");
    int goff[N];                                             // byte offset of the entry's source pixel
    uint32_t soff, vm;                                       // where entry 0's operand goes (entry e: e * NT * 16 on); entries inside the image
    const char* xb;
    uint4 raw[HALVES][N];
    __device__ __forceinline__ void prepare(const ConvArgs& a, int frame, int c_first, int ty, int tx, int H, int W, int ptid) {
        const int j = ptid & 7, pix0 = ptid >> 3;
        soff = (uint32_t)(pix0 * 128) + (IN_BF16 ? (uint32_t)((j ^ (pix0 & 7)) << 4) : (uint32_t)((((j >> 1) ^ (pix0 & 7)) << 4) + (j & 1) * 8));
        vm = 0u;
#pragma unroll
        for (int e = 0; e < N; ++e) {
            const int pix = (e * NT + ptid) >> 3, py = pix / PW, px = pix - py * PW;
            const int oy = ty + py - 1, ox = tx + px - 1;
            bool v = oy >= 0 && oy < H && ox >= 0 && ox < W && pix < NPIX;
            if (KIND == K1X1) v = v && py >= 1 && py <= TILE_H && px >= 1 && px <= TILE_W;
            vm |= (v ? 1u : 0u) << e;
            goff[e] = v ? (oy * W + ox) * a.Cin * ESZ : 0;
        }
        xb = (const char*)a.x + ((size_t)frame * H * W * a.Cin + c_first + j * NV) * ESZ;
    }
    __device__ __forceinline__ void load(int u, int h, int e) {
        if (vm >> e & 1u) raw[h][e] = convtile::ldg_stream(xb + (size_t)u * (64 * ESZ) + goff[e] + h * 128);
    }
    __device__ __forceinline__ void load_first() {
#pragma unroll
        for (int h = 0; h < HALVES; ++h)
#pragma unroll
            for (int e = 0; e < N; ++e) load(0, h, e);
    }
    __device__ __forceinline__ void transform(uint8_t* dst, int u, bool more, bool prologue, bool silu, const float* s_scale, const float* s_shift, int ptid) {
        const int j = ptid & 7;
#pragma unroll
        for (int h = 0; h < HALVES; ++h) {
            float sc[NV], sf[NV];
            if (prologue) {
                const int c = u * 64 + j * NV + h * 32;
#pragma unroll
                for (int i = 0; i < NV; i += 4) {
                    *(float4*)&sc[i] = *(const float4*)(s_scale + c + i);
                    *(float4*)&sf[i] = *(const float4*)(s_shift + c + i);
                }
            }
#pragma unroll
            for (int e = 0; e < N; ++e) {
                if (e == N - 1 && ((e * NT + ptid) >> 3) >= NPIX) break;
                uint32_t o[NV / 2];
#pragma unroll
                for (int i = 0; i < NV / 2; ++i) o[i] = 0u;
                if (vm >> e & 1u) {
                    float v[NV];
                    const uint32_t r[4] = {raw[h][e].x, raw[h][e].y, raw[h][e].z, raw[h][e].w};
#pragma unroll
                    for (int i = 0; i < NV; ++i)
                        v[i] = __uint_as_float(!IN_BF16 ? r[i & 3] : (i & 1) ? r[i >> 1] & 0xffff0000u : r[i >> 1] << 16);
                    if (more) load(u + 1, h, e);
                    if (prologue) {
#pragma unroll
                        for (int i = 0; i < NV; ++i) v[i] = fmaf(v[i], sc[i], sf[i]);
                        if (silu) {
#pragma unroll
                            for (int i = 0; i < NV; ++i) v[i] = fmaf(v[i], tanh_fast(v[i]), v[i]);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < NV / 2; ++i) o[i] = KIND == KPHASE ? pack_f16(v[2 * i], v[2 * i + 1]) : pack_bf16(v[2 * i], v[2 * i + 1]);
                }
                uint8_t* d = dst + (h ? soff ^ 64u : soff) + e * (NT * 16);
                if constexpr (IN_BF16) *(uint4*)d = make_uint4(o[0], o[1], o[2], o[3]);
                else *(uint2*)d = make_uint2(o[0], o[1]);
            }
        }
    }
};

// BN: output channels per cluster (16: the frame head).  KIND: 3x3, 1x1, or one output parity of the phase-collapsed
// upsampling convolution (2x2 taps of the source, fp16 operands; see conv_tc.cu).
template <int BN, int KIND, bool IN_BF16>
__global__ void __launch_bounds__(kThreads, 2)
conv_split_kernel(const ConvArgs a, const ConvSplitShape sh, const __grid_constant__ CUtensorMap tm_w,
                  const __grid_constant__ CUtensorMap tm_w2, const __grid_constant__ CUtensorMap tm_x2, unsigned int* status) {
    constexpr int TAPS = taps_of(KIND);
    constexpr int BST = BN * 128;                            // bytes of a weight stage
    constexpr int ROWS = TILE_H * TILE_W, CB = BN < 64 ? BN : 32, NB = BN / CB;       // a warp moves 32 rows x CB channels of the accumulator
    constexpr int ACC_COLS = BN < 32 ? 32 : BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int n_a = sh.n_a, n_b = sh.n_b, S = sh.splits;
    uint8_t* smem_a = smem;
    uint8_t* smem_b = smem + n_a * A_TILE_BYTES;
    // over the operand stages, once every MMA of the cluster is done: this CTA's partials [NB][ROWS][CB], and those of its
    // rows [S][NB][rows][CB]
    float* part = (float*)smem;
    float* rx = S > 1 ? part + ROWS * BN : part;
    float* s_scale = (float*)(smem + sh.tail_off);
    float* s_shift = s_scale + kMaxSliceC;
    SBars* bars = (SBars*)(s_shift + kMaxSliceC);
    static_assert(sizeof(SBars) <= 256, "barrier block");
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_ctarank();

    // ---- this cluster's item: (frame, tile, output parity, channel block); for KPHASE the tile grid is that of the source
    const int H = KIND == KPHASE ? a.Hs : a.H, W = KIND == KPHASE ? a.Ws : a.W;
    const int tiles_x = (W + TILE_W - 1) / TILE_W, tiles = tiles_x * ((H + TILE_H - 1) / TILE_H);
    const int nblk = (a.Cout + BN - 1) / BN;
    int item = (int)blockIdx.x / S;
    const int n0 = (item % nblk) * BN;
    item /= nblk;
    const int par = KIND == KPHASE ? (item & 3) : 0;
    if (KIND == KPHASE) item >>= 2;
    const int tile = item % tiles, frame = item / tiles;
    const int ty = (tile / tiles_x) * TILE_H, tx = (tile % tiles_x) * TILE_W;
    const int kchunks = a.Cin >> 6, kchunks2 = a.x2 ? (a.Cin2 >> 5) : 0;
    const int k0 = rank * kchunks / S, nk = (rank + 1) * kchunks / S - k0;           // chunks of this CTA
    const int q0 = rank * kchunks2 / S, nq = (rank + 1) * kchunks2 / S - q0;         // sub-chunks of the fused shortcut
    const int units = nk + nq, loads = nk * TAPS + nq;

    if (tid == 0) {
        for (int i = 0; i < n_a; ++i) { mbar_init(smem_u32(&bars->a_full[i]), 8); mbar_init(smem_u32(&bars->a_empty[i]), 1); }
        for (int i = 0; i < n_b; ++i) { mbar_init(smem_u32(&bars->b_full[i]), 1); mbar_init(smem_u32(&bars->b_empty[i]), 1); }
        mbar_init(smem_u32(&bars->acc_full), S);             // one commit from every CTA of the cluster
        mbar_init(smem_u32(&bars->rx_full), 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(smem_u32(&bars->rx_full), ROWS * BN * 4);  // this CTA's rows from all S partials
    }
    if (warp == 0) tmem_alloc(smem_u32(&bars->tmem_base), (uint32_t)ACC_COLS);
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
            for (int u = 0; u < units && ok; ++u) {
                const bool second = u >= nk;
                const int ntap = second ? 1 : TAPS;
#pragma unroll 1
                for (int tap = 0; tap < ntap; ++tap) {
                    if (issued >= n_b) ok = mbar_wait(smem_u32(&bars->b_empty[st]), ph ^ 1, abort_flag);
                    if (!ok) break;
                    const uint32_t full = smem_u32(&bars->b_full[st]), dst = smem_u32(smem_b + st * BST);
                    mbar_arrive_expect_tx(full, BST);
                    // row of the packed weights: [tap][Cout], or (phase form) [2 * parity + dy][128-channel block][half of it][dx][64]
                    const int row = KIND == KPHASE ? ((((2 * par + (tap >> 1)) * (a.Cout / 128) + n0 / 128) * 2 + ((n0 >> 6) & 1)) * 2 + (tap & 1)) * 64
                                                   : tap * sh.w_rows + n0;
                    if (second) tma_load_2d(dst, &tm_w2, (q0 + u - nk) * 32, n0, full);
                    else tma_load_2d(dst, &tm_w, (k0 + u) * 64, row, full);
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
        constexpr uint32_t idesc = KIND == KPHASE ? make_idesc_f16(128, BN) : make_idesc_bf16(128, BN);
        constexpr uint32_t idesc_tf32 = make_idesc_tf32(128, BN);
        const uint32_t a_hi = desc_hi(PW * 128, 2), d_hi = desc_hi(1024, 2);
        const uint32_t a_lo0 = desc_lo(smem_u32(smem_a)), b_lo0 = desc_lo(smem_u32(smem_b));
        uint32_t as = 0, aph = 0, bs = 0, bph = 0, acc = 0;
        int used = 0;                                        // a stage that no later load needs is not handed back
        auto wait_on = [&](uint64_t* b, uint32_t ph) {
            if (!mbar_try_wait(smem_u32(b), ph)) (void)mbar_wait(smem_u32(b), ph, abort_flag);
            tc_fence_after();
        };
        auto stage_done = [&] {
            if (++used + n_b <= loads) umma_commit_on(smem_u32(&bars->b_empty[bs]), lead);
            __syncwarp();
            if (++bs == (uint32_t)n_b) { bs = 0; bph ^= 1; }
        };
#pragma unroll 1
        for (int u = 0; u < units; ++u) {
            if (*abort_flag) break;
            wait_on(&bars->a_full[as], aph);
            const uint32_t a_st = a_lo0 + as * (uint32_t)(A_TILE_BYTES >> 4);
            if (BN == 64 && KIND == K3X3 && u >= nk) {       // shortcut sub-chunk: fp32 operands, four kind::tf32 MMAs of K = 8
                wait_on(&bars->b_full[bs], bph);
                const uint32_t b_lo = b_lo0 + bs * (uint32_t)(BST >> 4);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    umma_tf32_split_on(tmem, a_st + 2 * k, d_hi, b_lo + 2 * k, d_hi, idesc_tf32, acc, lead);
                    acc = 1u;
                }
                stage_done();
            } else {
                uint32_t a_lo = a_st + (KIND == K1X1 ? (uint32_t)((PW + 1) * 8) : KIND == KPHASE ? (uint32_t)(((par >> 1) * PW + (par & 1)) * 8) : 0u);
                constexpr int COLS = KIND == K3X3 ? 3 : (KIND == K1X1 ? 1 : 2);
                int kx = 0;
#pragma unroll 1
                for (int tap = 0; tap < TAPS; ++tap) {
                    wait_on(&bars->b_full[bs], bph);
                    const uint32_t b_lo = b_lo0 + bs * (uint32_t)(BST >> 4);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        umma_bf16_split_on(tmem, a_lo + 2 * k, a_hi, b_lo + 2 * k, d_hi, idesc, acc, lead);
                        acc = 1u;
                    }
                    stage_done();
                    if (++kx == COLS) { kx = 0; a_lo += (uint32_t)((PW - COLS + 1) * 8); } else a_lo += 8u;
                }
            }
            if (u + n_a < units) umma_commit_on(smem_u32(&bars->a_empty[as]), lead);
            __syncwarp();
            if (++as == (uint32_t)n_a) { as = 0; aph ^= 1; }
        }
        __syncwarp();
        cluster_wait();
        commit_to_cluster(smem_u32(&bars->acc_full), (uint16_t)((1u << S) - 1u), lead);
        __syncwarp();
    } else {
        // ------------------------------------------------ operand prologue
        const int ptid = tid - kProd0 * 32, pw = warp - kProd0;
        const bool prologue = a.scale != nullptr || a.in_rec != nullptr, silu = a.silu != 0;
        const int nch = nk * 64;
        const float half = silu ? 0.5f : 1.0f;               // SiLU is evaluated as h + h * tanh(h), h = v / 2
        Operand<KIND, IN_BF16, 8> op;
        op.prepare(a, frame, k0 * 64, ty, tx, H, W, ptid);
        InputStats stats;
        if (a.in_rec) stats.prepare(a, frame, k0 * 64, nch, pw, lane, s_scale, s_shift);
        if (pw == 0) touch_params(a, &bars->unused);
        griddep_wait();
        if (a.in_rec) stats.load(a, lane);
        uint32_t as = 0, aph = 0;
        bool ok = true;
        op.load_first();
#pragma unroll 1
        for (int u = 0; u < units; ++u) {
            const bool second = BN == 64 && KIND == K3X3 && u >= nk;
            uint8_t* dst = smem_a + as * A_TILE_BYTES;
            if (u == 0 && prologue) {
                if (a.in_rec) stats.finish(a, nch, lane, half, s_scale, s_shift);
                else
                    for (int c = ptid; c < nch; c += kProd) {
                        s_scale[c] = __ldcg(a.scale + (size_t)frame * a.Cin + k0 * 64 + c) * half;
                        s_shift[c] = __ldcg(a.shift + (size_t)frame * a.Cin + k0 * 64 + c) * half;
                    }
                named_barrier_sync(1, kProd);
            }
            if (u >= n_a) {
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->a_empty[as]), aph ^ 1, abort_flag));
                if (!ok) break;
            }
            if (second) {                                    // 16 x 8 pixels x 32 fp32 channels, as they lie in memory
                if (ptid == 0) {
                    mbar_expect_tx(smem_u32(&bars->a_full[as]), TILE_H * TILE_W * 128);
                    tma_load_4d(smem_u32(dst), &tm_x2, (q0 + u - nk) * 32, tx, ty, frame, smem_u32(&bars->a_full[as]));
                }
            } else {
                op.transform(dst, u, u + 1 < nk, prologue, silu, s_scale, s_shift, ptid);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars->a_full[as]));
            if (++as == (uint32_t)n_a) { as = 0; aph ^= 1; }
        }
        // ------------------------------------------------ exchange and epilogue: row R of the tile belongs to CTA R / rpo
        const int rpo_log2 = 7 - (__ffs(S) - 1), rpo = 1 << rpo_log2;                 // (S is a power of two)
        static_assert(ROWS == 128, "rows of a tile");
        auto exchange = [&] {
            (void)mbar_wait(smem_u32(&bars->acc_full), 0, abort_flag);       // every CTA of the cluster is done with its operands
            tc_fence_after();
            __syncwarp();
            cluster_wait();
            const int cb = BN < 64 ? 0 : pw >> 2, R0 = (warp & 3) * 32;
            float* row = part + (cb * ROWS + R0 + lane) * CB;
            const uint32_t tacc = tmem + (uint32_t)(cb * CB) + ((uint32_t)R0 << 16);
            const bool moves = BN >= 64 || pw < 4;
            uint32_t r[CB];
            if constexpr (BN < 64) tmem_ld16(tacc, r);
            else tmem_ld32(tacc, r);
            tmem_ld_wait();
            if (moves) {
#pragma unroll
                for (int c = 0; c < CB / 4; ++c) *(uint4*)(row + exchange_piece<BN>(lane, c) * 4) = make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
            }
            tc_fence_before();
            if (S > 1) {                                     // each warp sends what it has written: its owners' rows lie together
                fence_proxy_async_smem();
                __syncwarp();
                const int n_log2 = min(rpo_log2, 5), n = 1 << n_log2, R = R0 + lane * n, owner = R >> rpo_log2;
                if (moves && lane < 32 >> n_log2)
                    copy_to_peer(map_to_cta(smem_u32(rx + ((rank * NB + cb) * rpo + R - owner * rpo) * CB), (uint32_t)owner), smem_u32(part + (cb * ROWS + R) * CB),
                                 (uint32_t)(n * CB * 4), map_to_cta(smem_u32(&bars->rx_full), (uint32_t)owner));
                __syncwarp();
                (void)wait_cluster(smem_u32(&bars->rx_full), 0, abort_flag);
            } else {
                named_barrier_sync(1, kProd);
            }
            __syncwarp();
            cluster_arrive();                                // what is sent to this CTA has landed
        };
        finish_rows<BN, 2>(a, [&](int s, int local, int c) { return rx + ((s * NB + c / (CB / 4)) * rpo + local) * CB + exchange_piece<BN>(local, c % (CB / 4)) * 4; }, S, rpo, ptid, frame, n0, KIND == KPHASE ? 2 * H : H, KIND == KPHASE ? 2 * W : W,
                        (KIND == KPHASE ? tile * 4 + par : tile) * S + rank,
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
    cluster_wait();                                          // the sources of this CTA's copies may go; its accumulator has been read
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)ACC_COLS);
    }
    if (tid == kProd0 * 32 && bars->abort_flag && status) {
        if (atomicCAS(status, 0u, kStatusConvTimeout) == 0u) {
            status[1] = blockIdx.x;
            status[2] = (uint32_t)BN;
        }
    }
}

// ---- the same on pairs of CTAs
// Where 64-channel blocks would stream the weights too often, a pair of CTAs takes two tiles x 256 output channels as one
// tcgen05.mma.cta_group::2 (M = 256): a tap's weights come from L2 once for both tiles, and each CTA's shared memory holds
// and feeds half of them.  S pairs share K; the exchange is between the CTAs of the same tile.  The pair's even CTA issues;
// all "full" barriers are its own.
constexpr int kPairBN = 256, kPairWarps = 16, kPairThreads = (kProd0 + kPairWarps) * 32, kPairSmemMax = 227 * 1024, kPairSplits = 2;

// arrives, once the pair's MMAs issued so far have completed, on the barrier at this offset in every CTA of `mask`
__device__ __forceinline__ void commit2_to_cluster(uint32_t bar, uint16_t mask, uint32_t on) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n"
                 "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n"
                 ::"r"(bar), "h"(mask), "r"(on) : "memory");
}

template <bool IN_BF16>
__global__ void __launch_bounds__(kPairThreads, 1)
conv_pair_kernel(const ConvArgs a, const ConvSplitShape sh, const __grid_constant__ CUtensorMap tm_w, unsigned int* status) {
    constexpr int TAPS = 9, BN = kPairBN, BST = BN / 2 * 128, ROWS = TILE_H * TILE_W, CB = 64, NT = kPairWarps * 32, S = kPairSplits, RPO = ROWS / S;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int n_a = sh.n_a, n_b = sh.n_b;
    uint8_t* smem_a = smem;
    uint8_t* smem_b = smem + n_a * A_TILE_BYTES;
    // over the operand stages, once every MMA of the cluster is done: this CTA's partials [4][ROWS][CB], and the other CTA's
    // of its rows [4][RPO][CB]
    float* part = (float*)smem;
    float* rx = part + ROWS * BN;
    float* s_scale = (float*)(smem + sh.tail_off);
    float* s_shift = s_scale + kMaxSliceC;
    SBars* bars = (SBars*)(s_shift + kMaxSliceC);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_ctarank(), half = rank & 1, kp = rank >> 1, lead_cta = rank & ~1;
    const int H = a.H, W = a.W;
    const int tiles_x = (W + TILE_W - 1) / TILE_W, tiles = tiles_x * ((H + TILE_H - 1) / TILE_H), groups = (tiles + 1) / 2;
    const int nblk = a.Cout / BN;
    int item = (int)blockIdx.x / (2 * S);
    const int n0 = (item % nblk) * BN;
    item /= nblk;
    const int tile = (item % groups) * 2 + half, frame = item / groups;
    const int ty = tile / tiles_x * TILE_H, tx = tile % tiles_x * TILE_W;            // (beyond the last tile: below the image, nothing out)
    const int kchunks = a.Cin >> 6, k0 = kp * kchunks / S, nk = (kp + 1) * kchunks / S - k0;

    if (tid == 0) {
        for (int i = 0; i < n_a; ++i) { mbar_init(smem_u32(&bars->a_full[i]), 2 * kPairWarps); mbar_init(smem_u32(&bars->a_empty[i]), 1); }
        for (int i = 0; i < n_b; ++i) { mbar_init(smem_u32(&bars->b_full[i]), 2); mbar_init(smem_u32(&bars->b_empty[i]), 1); }
        mbar_init(smem_u32(&bars->acc_full), S);             // one commit from every pair of the cluster
        mbar_init(smem_u32(&bars->rx_full), 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(smem_u32(&bars->rx_full), RPO * BN * 4);                  // this CTA's rows from the other partial
    }
    if (warp == 0) tmem_alloc2(smem_u32(&bars->tmem_base), (uint32_t)BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_arrive();
    cluster_wait();                                          // every CTA's barriers exist before anyone signals across
    const uint32_t tmem = bars->tmem_base;
    griddep_launch();

    if (warp == 1) {
        // ------------------------------------------------ this CTA's half of the weights (they do not depend on the kernel before)
        if (lane == 0) {
            uint32_t st = 0, ph = 0;
            int issued = 0;
            bool ok = true;
            for (int u = 0; u < nk && ok; ++u) {
#pragma unroll 1
                for (int tap = 0; tap < TAPS; ++tap) {
                    if (issued >= n_b) ok = mbar_wait(smem_u32(&bars->b_empty[st]), ph ^ 1, abort_flag);
                    if (!ok) break;
                    const uint32_t full = map_to_cta(smem_u32(&bars->b_full[st]), lead_cta);
                    mbar_arrive_expect_tx_cluster(full, BST);
                    tma_load_2d_pair(smem_u32(smem_b + st * BST), &tm_w, (k0 + u) * 64, tap * a.Cout + n0 + half * (BN / 2), full);
                    ++issued;
                    if (++st == (uint32_t)n_b) { st = 0; ph ^= 1; }
                }
            }
            // what a pair that gave up has on its way lands before anybody may leave (the last arrival below); both halves are
            // counted on the even CTA's barriers
            (void)mbar_wait(smem_u32(&bars->acc_full), 0, abort_flag);
            if (half == 0 && *abort_flag) land_loads(bars->b_full, n_b, issued);
        }
    } else if (warp == 0) {
        // ------------------------------------------------ MMA issue (warp-uniform, predicated on one elected lane)
        if (half == 0) {
            const uint32_t lead = elect_one();
            constexpr uint32_t idesc = make_idesc_bf16(256, BN);
            const uint32_t a_hi = desc_hi(PW * 128, 2), d_hi = desc_hi(1024, 2);
            const uint32_t a_lo0 = desc_lo(smem_u32(smem_a)), b_lo0 = desc_lo(smem_u32(smem_b));
            const uint16_t pair_mask = (uint16_t)(3u << rank), all = (uint16_t)((1u << (2 * S)) - 1u);
            const int loads = nk * TAPS;
            uint32_t as = 0, aph = 0, bs = 0, bph = 0, acc = 0;
            int used = 0;                                    // a stage that no later load needs is not handed back
            auto wait_on = [&](uint64_t* b, uint32_t ph) {
                if (!mbar_try_wait(smem_u32(b), ph)) (void)mbar_wait(smem_u32(b), ph, abort_flag);
                tc_fence_after();
            };
#pragma unroll 1
            for (int u = 0; u < nk; ++u) {
                if (*abort_flag) break;
                wait_on(&bars->a_full[as], aph);
                uint32_t a_lo = a_lo0 + as * (uint32_t)(A_TILE_BYTES >> 4);
                int kx = 0;
#pragma unroll 1
                for (int tap = 0; tap < TAPS; ++tap) {
                    wait_on(&bars->b_full[bs], bph);
                    const uint32_t b_lo = b_lo0 + bs * (uint32_t)(BST >> 4);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        umma2_bf16_split_on(tmem, a_lo + 2 * k, a_hi, b_lo + 2 * k, d_hi, idesc, acc, lead);
                        acc = 1u;
                    }
                    if (++used + n_b <= loads) commit2_to_cluster(smem_u32(&bars->b_empty[bs]), pair_mask, lead);
                    __syncwarp();
                    if (++bs == (uint32_t)n_b) { bs = 0; bph ^= 1; }
                    if (++kx == 3) { kx = 0; a_lo += (uint32_t)((PW - 2) * 8); } else a_lo += 8u;
                }
                if (u + n_a < nk) commit2_to_cluster(smem_u32(&bars->a_empty[as]), pair_mask, lead);
                __syncwarp();
                if (++as == (uint32_t)n_a) { as = 0; aph ^= 1; }
            }
            __syncwarp();
            commit2_to_cluster(smem_u32(&bars->acc_full), all, lead);
            __syncwarp();
        }
    } else {
        // ------------------------------------------------ operand prologue
        const int ptid = tid - kProd0 * 32, pw = warp - kProd0;
        const bool prologue = a.scale != nullptr || a.in_rec != nullptr, silu = a.silu != 0;
        const int nch = nk * 64;
        const float scale = silu ? 0.5f : 1.0f;              // SiLU is evaluated as h + h * tanh(h), h = v / 2
        Operand<K3X3, IN_BF16, kPairWarps> op;
        op.prepare(a, frame, k0 * 64, ty, tx, H, W, ptid);
        InputStatsOf<kPairWarps, 4> stats;
        if (a.in_rec) stats.prepare(a, frame, k0 * 64, nch, pw, lane, s_scale, s_shift);
        if (pw == 0) touch_params(a, &bars->unused);
        griddep_wait();
        if (a.in_rec) stats.load(a, lane);
        op.load_first();
        if (prologue) {
            if (a.in_rec) {
                stats.finish(a, nch, lane, scale, s_scale, s_shift);
            } else {
                for (int c = ptid; c < nch; c += NT) {
                    s_scale[c] = __ldcg(a.scale + (size_t)frame * a.Cin + k0 * 64 + c) * scale;
                    s_shift[c] = __ldcg(a.shift + (size_t)frame * a.Cin + k0 * 64 + c) * scale;
                }
            }
            named_barrier_sync(1, NT);
        }
        uint32_t as = 0, aph = 0;
#pragma unroll 1
        for (int u = 0; u < nk; ++u) {
            if (u >= n_a && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->a_empty[as]), aph ^ 1, abort_flag))) break;
            op.transform(smem_a + as * A_TILE_BYTES, u, u + 1 < nk, prologue, silu, s_scale, s_shift, ptid);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bars->a_full[as]), lead_cta));
            if (++as == (uint32_t)n_a) { as = 0; aph ^= 1; }
        }
        // ------------------------------------------------ exchange and epilogue: row R of the tile belongs to part R / rpo of K,
        // and to eight of the sixteen warps
        constexpr int rows = RPO / 2;
        const int first = (pw >> 3) * rows;
        auto exchange = [&] {
            (void)mbar_wait(smem_u32(&bars->acc_full), 0, abort_flag);       // every CTA of the cluster is done with its operands
            tc_fence_after();
            __syncwarp();
            const int cb = pw >> 2, R0 = (warp & 3) * 32, owner = R0 / RPO;
            float* row = part + (cb * ROWS + R0 + lane) * CB;
#pragma unroll 1
            for (int p = 0; p < CB; p += 32) {
                uint32_t r[32];
                tmem_ld32(tmem + (uint32_t)(cb * CB + p) + ((uint32_t)R0 << 16), r);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 8; ++c) *(uint4*)(row + exchange_piece<BN>(lane, (p >> 2) + c) * 4) = make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
            }
            tc_fence_before();
            fence_proxy_async_smem();
            __syncwarp();
            if (owner != kp && lane == 0) {
                const uint32_t peer = (uint32_t)(owner * 2 + half);
                copy_to_peer(map_to_cta(smem_u32(rx + (cb * RPO + R0 - owner * RPO) * CB), peer), smem_u32(part + (cb * ROWS + R0) * CB), 32 * CB * 4,
                             map_to_cta(smem_u32(&bars->rx_full), peer));
            }
            named_barrier_sync(1, NT);                       // this CTA's own share of its rows
            (void)wait_cluster(smem_u32(&bars->rx_full), 0, abort_flag);
            __syncwarp();
            cluster_arrive();                                // what is sent to this CTA has landed
        };
        finish_rows<BN, 4>(a, [&](int s, int local, int c) {
                                    const int b = c / (CB / 4), R = first + local;
                                    return (s == kp ? part + (b * ROWS + kp * RPO + R) * CB : rx + (b * RPO + R) * CB) + exchange_piece<BN>(R, c % (CB / 4)) * 4;
                                }, S, rows,
                                ptid & 255, frame, n0, H, W, (tile * S + kp) * 2 + (pw >> 3),
                                [&](int local, int& oy, int& ox) -> bool {
                                    const int R = kp * RPO + first + local;
                                    oy = ty + (R >> 3);
                                    ox = tx + (R & 7);
                                    return oy < H && ox < W;
                                },
                                exchange);
    }
    __syncwarp();
    if (warp < kProd0) cluster_arrive();
    cluster_wait();                                          // the sources of this CTA's copies may go; the pair's accumulators have been read
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc2(tmem, (uint32_t)BN);
    }
    if (tid == kProd0 * 32 && bars->abort_flag && status) {
        if (atomicCAS(status, 0u, kStatusConvTimeout) == 0u) {
            status[1] = blockIdx.x;
            status[2] = (uint32_t)BN;
        }
    }
}

int kind_of(const ConvArgs& a) { return a.upsample == 2 ? KPHASE : (a.ksize == 1 ? K1X1 : K3X3); }
int tiles_of(const ConvArgs& a) {
    const int h = a.upsample == 2 ? a.Hs : a.H, w = a.upsample == 2 ? a.Ws : a.W;
    return ((w + TILE_W - 1) / TILE_W) * ((h + TILE_H - 1) / TILE_H);
}

template <int BN, int KIND, bool IB>
cudaError_t launch_one(const ConvArgs& a, const ConvSplitPlan& p, unsigned int* status, cudaStream_t s) {
    const long long ctas = (long long)tiles_of(a) * ((a.Cout + BN - 1) / BN) * (KIND == KPHASE ? 4 : 1) * a.B * p.shape.splits;
    return launch_clusters<conv_split_kernel<BN, KIND, IB>>({ctas, kThreads, p.smem, kSplitSmemMax, p.shape.splits}, s, a, p.shape, *(const CUtensorMap*)p.tmap,
                                                            *(const CUtensorMap*)p.tmap2, *(const CUtensorMap*)p.tmap_x2, status);
}

template <bool IB>
cudaError_t launch_pair(const ConvArgs& a, const ConvSplitPlan& p, unsigned int* status, cudaStream_t s) {
    const long long ctas = (long long)(tiles_of(a) + 1) / 2 * (a.Cout / kPairBN) * a.B * 2 * p.shape.splits;
    return launch_clusters<conv_pair_kernel<IB>>({ctas, kPairThreads, p.smem, kPairSmemMax, 2 * p.shape.splits}, s, a, p.shape, *(const CUtensorMap*)p.tmap, status);
}

}  // namespace

// (The upsampling form and the frame head read the residual stream: fp32 input only.)
bool conv_split_supported(const ConvArgs& a) {
    return conv_tc_supported(a) && a.upsample != 1 && !(a.residual && a.out_dtype != VD_F32) &&
           !(a.in_dtype == VD_BF16 && (a.upsample == 2 || a.Cout % 128 != 0));
}

int conv_split_slots(const ConvArgs& a, const ConvSplitPlan& p, int groups) {
    if (p.bn == kPairBN) return (tiles_of(a) + 1) / 2 * 2 * p.shape.splits * 2 * rec_parts(p.bn, a.Cout / groups);
    return tiles_of(a) * (a.upsample == 2 ? 4 : 1) * p.shape.splits * rec_parts(p.bn, a.Cout / groups);
}

// Layers whose CTAs, with K divided among up to 8 of them, stay within two per SM and walk 128 input channels each at most.
// Measured with both (one B200): up to there a layer with its normalisation takes 8-12 us against 25-45 on conv_tc.cu;
// with 512 channels per CTA (256x256 frame, 64x64 level) this kernel's narrow channel blocks stream the weights four
// times as often as conv_tc.cu's, and a 424x296 frame took 1.73 instead of 1.57 ms.
// Beyond, 3x3 layers run on pairs with K in two as long as the clusters of four fit the chip at once (33 of them; from 10, where
// 64-channel blocks no longer do): a layer with its normalisation 22 us against 40 on conv_tc.cu (64x64 and 37x53 pixels, 512
// channels, 32 and 22 pairs); 256x256 frame 1016 -> 957 us, 424x296 1534 -> 1455; with 10, 12 and 14 pairs at the second level
// (160x128, 192x128, 224x128 frames) 790 -> 736, 810 -> 755, 802 -> 744.  Pairs without the division (60x90, 74x106) gain
// nothing over conv_tc.cu.  (296 and 132: two CTAs and 0.9 CTAs per SM of 148; on fewer SMs the layers take more waves.)
bool conv_split_choose(const ConvArgs& a, ConvSplitPlan* p) {
    p->valid = 0;
    if (!conv_split_supported(a)) return false;
    const int kind = kind_of(a), kchunks = a.Cin / 64, taps = taps_of(kind);
    const bool head = a.Cout % 128 != 0;
    const int bn = head ? 16 : 64;
    const long long ctas = (long long)tiles_of(a) * ((a.Cout + bn - 1) / bn) * (kind == KPHASE ? 4 : 1) * std::max(a.B, 1);
    int s = 1;
    while (s < 8 && 2 * s <= kchunks && ctas * 2 * s <= 296) s *= 2;
    if (ctas * s > 296 || kchunks / s > 2) {
        if (kind != K3X3 || a.x2 || a.Cout % kPairBN != 0) return false;
        const long long pairs = (long long)(tiles_of(a) + 1) / 2 * (a.Cout / kPairBN) * std::max(a.B, 1);
        if (kchunks < kPairSplits || 2 * kPairSplits * pairs > 132) return false;
        s = kPairSplits;
        const int nk = (kchunks + s - 1) / s, rows = TILE_H * TILE_W;
        if (nk * 64 > kMaxSliceC) return false;
        const int na = std::min(nk, kMaxA), a_bytes = na * A_TILE_BYTES, bst = kPairBN / 2 * 128;
        const int nb = std::min(std::min(nk * taps, kMaxB), (kPairSmemMax - 1024 - kTailBytes - a_bytes) / bst);
        const int ops = std::max(a_bytes + nb * bst, (rows + rows / s * (s - 1)) * kPairBN * 4);
        if (nb < 1 || ops + kTailBytes + 1024 > kPairSmemMax) return false;
        p->bn = kPairBN;
        p->shape = ConvSplitShape{s, na, nb, ops, a.Cout};
        p->smem = ops + kTailBytes + 1024;
        return true;
    }
    // stages: as many as let two CTAs share an SM; a CTA with one unit needs one operand stage only
    const int nk = (kchunks + s - 1) / s, nq = a.x2 ? (a.Cin2 / 32 + s - 1) / s : 0;
    const int na = std::min(nk + nq, kMaxA), a_bytes = na * A_TILE_BYTES, bst = bn * 128;
    const int nb = std::min(std::min(nk * taps + nq, kMaxB), (kSplitSmemMax - 1024 - kTailBytes - a_bytes) / bst);
    const int ops = (std::max(a_bytes + nb * bst, (s > 1 ? 2 : 1) * TILE_H * TILE_W * bn * 4) + 15) / 16 * 16;
    if (ops + kTailBytes + 1024 > kSplitSmemMax) return false;
    p->bn = bn;
    p->shape = ConvSplitShape{s, na, nb, ops, head ? 16 : a.Cout};
    p->smem = ops + kTailBytes + 1024;
    return true;
}

cudaError_t conv_split_prepare(const ConvArgs& a, ConvSplitPlan* p) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const int rows = a.upsample == 2 ? 16 * a.Cout : a.ksize * a.ksize * p->shape.w_rows;
    const cuuint64_t wd[2] = {(cuuint64_t)a.Cin, (cuuint64_t)rows};
    const cuuint64_t ws[1] = {(cuuint64_t)a.Cin * 2};
    const cuuint32_t wb[2] = {64, (cuuint32_t)(p->bn == kPairBN ? kPairBN / 2 : p->bn)};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    if (enc((CUtensorMap*)p->tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(a.w), wd, ws, wb, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    memcpy(p->tmap2, p->tmap, sizeof(p->tmap));
    memcpy(p->tmap_x2, p->tmap, sizeof(p->tmap));
    if (a.x2) {
        const cuuint64_t d2[2] = {(cuuint64_t)a.Cin2, (cuuint64_t)a.Cout};
        const cuuint64_t s2[1] = {(cuuint64_t)a.Cin2 * 4};
        const cuuint32_t b2[2] = {32, (cuuint32_t)p->bn};
        if (enc((CUtensorMap*)p->tmap2, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(a.w2), d2, s2, b2, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        const cuuint64_t xd[4] = {(cuuint64_t)a.Cin2, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)std::max(a.B, 1)};
        const cuuint64_t xs[3] = {(cuuint64_t)a.Cin2 * 4, (cuuint64_t)a.W * a.Cin2 * 4, (cuuint64_t)a.H * a.W * a.Cin2 * 4};
        const cuuint32_t xb[4] = {32, (cuuint32_t)TILE_W, (cuuint32_t)TILE_H, 1};
        if (enc((CUtensorMap*)p->tmap_x2, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(a.x2), xd, xs, xb, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    p->batch = a.B;
    p->valid = 1;
    return cudaSuccess;
}

// f(Build<...>) for the build that the plan takes
namespace {
template <int BN, int KIND, bool IB> struct Build {
    static cudaError_t launch(const ConvArgs& a, const ConvSplitPlan& p, unsigned int* status, cudaStream_t s) { return launch_one<BN, KIND, IB>(a, p, status, s); }
    static bool fits(const ConvSplitPlan& p) { return clusters_fit<conv_split_kernel<BN, KIND, IB>>(kThreads, kSplitSmemMax, p.shape.splits); }
};
template <bool IB> struct PairBuild {
    static cudaError_t launch(const ConvArgs& a, const ConvSplitPlan& p, unsigned int* status, cudaStream_t s) { return launch_pair<IB>(a, p, status, s); }
    static bool fits(const ConvSplitPlan& p) { return clusters_fit<conv_pair_kernel<IB>>(kPairThreads, kPairSmemMax, 2 * p.shape.splits); }
};
template <class F> auto with_build(const ConvArgs& a, const ConvSplitPlan& p, F f) {
    const bool ib = a.in_dtype == VD_BF16;
    const int kind = kind_of(a);
    if (p.bn == kPairBN) return ib ? f(PairBuild<true>()) : f(PairBuild<false>());
    if (p.bn == 16) return f(Build<16, K3X3, false>());
    if (kind == K3X3) return ib ? f(Build<64, K3X3, true>()) : f(Build<64, K3X3, false>());
    if (kind == K1X1) return ib ? f(Build<64, K1X1, true>()) : f(Build<64, K1X1, false>());
    return f(Build<64, KPHASE, false>());
}
}  // namespace

bool conv_split_fits(const ConvArgs& a, const ConvSplitPlan& p) {
    return with_build(a, p, [&](auto build) { return build.fits(p); });
}

int conv_split_cluster(const ConvSplitPlan& p) { return p.shape.splits * (p.bn == kPairBN ? 2 : 1); }

cudaError_t launch_conv_split(const ConvArgs& a, const ConvSplitPlan& p, unsigned int* status, cudaStream_t s) {
    if (!p.valid || a.B > p.batch) return cudaErrorInvalidValue;
    if (a.in_rec && !rec_groups_ok(a.Cin, a.in_G)) return cudaErrorInvalidValue;
    if (a.out_rec && !rec_groups_ok(a.Cout, a.out_G)) return cudaErrorInvalidValue;
    return with_build(a, p, [&](auto build) { return build.launch(a, p, status, s); });
}

}  // namespace vd
