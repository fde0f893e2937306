// Fused single-head attention on tcgen05/TMEM for the decoder's mid block (C = 512 channels):
//   o[t,:] = sum_u softmax_u(scale * q[t,:].k[u,:]) v[u,:]
// A pair of CTAs (tcgen05.mma.cta_group::2, M = 128) owns 128 queries, 64 per CTA, and all 512 channels of their output:
// in this shape an accumulator of N columns takes N/2 columns of each CTA's tensor memory (lanes 0-63: the CTA's 64 rows
// and the first N/2 columns, lanes 64-127: the same rows and the others), so 512 channels take 256 columns and two score
// tiles of 256 keys the other 256.  Per 256-key tile:
//   S = Q K^T      Q stays in shared memory; each CTA loads half of every K chunk, the pair's tensor cores read both halves
//   softmax        eight warps, four threads per query row (64 keys each): running maximum with lazy rescaling of the
//                  output accumulator, exp2 in fp32, row sums in fp32, P rounded to bf16 and written to shared memory in
//                  the swizzled K-major operand layout
//   O += P V       V is consumed transposed ([channel][token], produced by a small transpose kernel), half per CTA
// The tensor core works on the next tile's scores while the softmax warps are busy.  The N x N score matrix never exists
// in memory.  Where the query tiles leave SMs idle the keys are divided too: `splits` pairs form a cluster, each takes its
// share of the key tiles, and their outputs meet in distributed shared memory, added in a fixed order.
// What bounds it: 256 KB of K and V come from L2 per tile and CTA for 4096 tensor cycles.  Against one CTA per 128 queries and
// half of the channels, which computes the scores twice and reads Q anew for every key tile (us, one B200, with the transpose, the
// same call again and again): 1024 tokens 30.8 -> 22.5, 1961 51.3 -> 28.7, 5400 117.9 -> 71.7, eight times 5400 753 -> 404, two times
// 14400 1379 -> 724, which is 1173 TFLOP/s, 73 % of the measured bf16 peak.  Within decodes that hold the GPU at its power cap:
// eight times 5400 878 -> 509, two times 14400 1611 -> 806.
// Every wait is bounded (see tc_common.cuh).
#include <algorithm>
#include <mutex>

#include "conv_cluster.cuh"
#include "tc_common.cuh"
#include "tc_pair.cuh"
#include "vd_internal.h"

namespace vd {

namespace {

using namespace tc;

constexpr int CH = 512, BQ = 128, ROWS = 64, BKV = 256, CHUNK = 64;      // ROWS: queries of one CTA
constexpr int QK_CHUNKS = CH / CHUNK;                        // 64-channel chunks of a score tile: two a stage
// A stage is two boxes (K: 128 keys x 64 channels; V: 128 channels x 64 keys, of either half of the channels), eight MMAs: a
// wait, four MMAs and a commit to both CTAs cost the issuing warp more than the 256 cycles they take (5400 tokens, three pairs
// per query tile: 89 us with half the stage, 79 with this; two times 14400: 952 and 806)
constexpr int STAGES = 4, BOX_BYTES = 128 * CHUNK * 2, STAGE_BYTES = 2 * BOX_BYTES;
constexpr int Q_BYTES = ROWS * CH * 2, P_BYTES = ROWS * BKV * 2, BLOCK_BYTES = ROWS * 128;   // BLOCK: 64 rows x 64 columns of Q or P
constexpr int SOFTMAX_WARPS = 8, LOAD_WARP = 8, MMA_WARP = 9;
constexpr int NUM_THREADS = 10 * 32;
constexpr float RESCALE_THRESHOLD = 8.0f;                    // log2 units: accumulators may grow by 2^8
constexpr int kMaxSplits = 4;                                // pairs of a cluster (eight CTAs)

struct Bars {
    uint64_t q_full, full[STAGES], empty[STAGES];
    uint64_t s_full[2], s_free[2];
    uint64_t p_full, pv_done, drained;
    uint32_t tmem_base, abort_flag;
};
constexpr int RED_BYTES = 4 * ROWS * 4;                      // what the four threads of a row tell one another
constexpr int SMEM_TOTAL = Q_BYTES + P_BYTES + STAGES * STAGE_BYTES + RED_BYTES + 256 + 1024;
static_assert(sizeof(Bars) <= 256 && SMEM_TOTAL <= 232448, "shared memory of one CTA");
static_assert(STAGES * STAGE_BYTES >= ROWS * CH * 4, "a CTA's output fits the stages");

struct AttnTcParams {
    void* o;
    int B, T, ld_o, splits;
    float scale_log2;        // scale * log2(e)
};

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// a CTA's unfinished output in its stages: 16-byte piece `piece` (four channels) of a row; eight rows of a piece lie on distinct banks
__device__ __forceinline__ uint32_t dump_at(int row, int piece) { return (uint32_t)(row * (CH * 4) + ((piece ^ (row & 7)) << 4)); }
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_cluster_f2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

__global__ void __launch_bounds__(NUM_THREADS, 1)
attn_tc_kernel(const AttnTcParams a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_vt, unsigned int* status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* smem_q = smem;
    uint8_t* smem_p = smem + Q_BYTES;
    uint8_t* smem_st = smem_p + P_BYTES;
    float* s_red = (float*)(smem_st + STAGES * STAGE_BYTES);         // [4][ROWS]; at the end (reference, sum) per row
    Bars* bars = (Bars*)((uint8_t*)s_red + RED_BYTES);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t crank = cluster_ctarank(), rank = crank & 1u, lead_cta = crank & ~1u;
    const int split = (int)(crank >> 1);
    const int q_tiles = (a.T + BQ - 1) / BQ, cid = (int)blockIdx.x / (2 * a.splits);
    const int b = cid / q_tiles, q0 = (cid - b * q_tiles) * BQ + (int)rank * ROWS;
    const int ntiles = (a.T + BKV - 1) / BKV;
    const int j0 = ntiles * split / a.splits, j1 = ntiles * (split + 1) / a.splits;    // this pair's key tiles (splits <= ntiles)

    if (tid == 0) {
        // the leader's "full", "free" and P barriers collect the arrivals of both CTAs of the pair; commits go to both
        mbar_init(smem_u32(&bars->q_full), 2);
        for (int i = 0; i < STAGES; ++i) { mbar_init(smem_u32(&bars->full[i]), 2); mbar_init(smem_u32(&bars->empty[i]), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&bars->s_full[i]), 1); mbar_init(smem_u32(&bars->s_free[i]), 2 * SOFTMAX_WARPS); }
        mbar_init(smem_u32(&bars->p_full), 2 * SOFTMAX_WARPS);
        mbar_init(smem_u32(&bars->pv_done), 1);
        mbar_init(smem_u32(&bars->drained), 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
    }
    if (warp == MMA_WARP) tmem_alloc2(smem_u32(&bars->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                      // every CTA's barriers exist before anyone signals across
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base, tmem_s = tmem + 256;      // O: 2 x 128 columns, S: 2 x 128
    auto leader_bar = [&](uint64_t* p) { return map_to_cta(smem_u32(p), lead_cta); };
    griddep_launch();            // the next kernel may set itself up from here on
    if (warp != MMA_WARP) griddep_wait();    // every role but the MMA issue loop touches activations of earlier kernels

    const int quarter = warp & 3, kb = (quarter >> 1) * 2 + (warp >> 2), row = (quarter & 1) * 32 + lane;
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    if (warp < SOFTMAX_WARPS) {
        // ------------------------------------------------------------ softmax warps
        // A thread holds 64 keys (block kb of the tile) of one query row; the row's four threads sit in the warps with the
        // same (quarter & 1), which share a named barrier.
        float* red = s_red + row;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16, half_cols = (uint32_t)(warp >> 2) * 64u;
        // After a wait gave up a warp walks on over whatever is there: the four warps of a row meet at their barriers however each
        // of them learns of it, and nothing of it is written in the end.
        for (int j = j0; j < j1; ++j) {
            const int i = j - j0, buf = i & 1;
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->s_full[buf]), (i >> 1) & 1, abort_flag)) && ok;
            tc_fence_after();
            uint32_t r0[32], r1[32];
            tmem_ld32(tmem_s + lane_base + (uint32_t)buf * 128u + half_cols, r0);
            tmem_ld32(tmem_s + lane_base + (uint32_t)buf * 128u + half_cols + 32u, r1);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_relaxed(leader_bar(&bars->s_free[buf]));   // the scores are in registers
            const int kvalid = min(max(a.T - j * BKV - kb * 64, 0), 64);       // keys of this block that exist
            float tmax = -INFINITY;
            if (kvalid == 64) {
                float t0 = -INFINITY, t1 = -INFINITY;
#pragma unroll
                for (int q = 0; q < 32; ++q) {
                    t0 = fmaxf(t0, __uint_as_float(r0[q]) * a.scale_log2);
                    t1 = fmaxf(t1, __uint_as_float(r1[q]) * a.scale_log2);
                }
                tmax = fmaxf(t0, t1);
            } else {
#pragma unroll
                for (int q = 0; q < 32; ++q) {
                    if (q < kvalid) tmax = fmaxf(tmax, __uint_as_float(r0[q]) * a.scale_log2);
                    if (q + 32 < kvalid) tmax = fmaxf(tmax, __uint_as_float(r1[q]) * a.scale_log2);
                }
            }
            red[kb * ROWS] = tmax;
            named_barrier_sync(1 + (quarter & 1), SOFTMAX_WARPS * 16);
            tmax = fmaxf(fmaxf(red[0], red[ROWS]), fmaxf(red[2 * ROWS], red[3 * ROWS]));
            named_barrier_sync(1 + (quarter & 1), SOFTMAX_WARPS * 16);      // (the next tile writes again)
            // lazy rescale: keep the old reference unless the maximum grew by more than the threshold
            float factor = 1.f;
            const bool grow = tmax > m_ref + RESCALE_THRESHOLD;
            if (grow) {
                factor = ex2(m_ref - tmax);                        // 0 at the first tile (m_ref = -inf)
                m_ref = tmax;
                l *= factor;
            }
            // p = 2^(s - m_ref), row sum, bf16
            uint32_t pk[32];
            {
                float l0 = 0.f, l1 = 0.f;
#pragma unroll
                for (int q = 0; q < 32; q += 2) {
                    float e0 = ex2(fmaf(__uint_as_float(r0[q]), a.scale_log2, -m_ref)), e1 = ex2(fmaf(__uint_as_float(r0[q + 1]), a.scale_log2, -m_ref));
                    float f0 = ex2(fmaf(__uint_as_float(r1[q]), a.scale_log2, -m_ref)), f1 = ex2(fmaf(__uint_as_float(r1[q + 1]), a.scale_log2, -m_ref));
                    if (kvalid != 64) {
                        e0 = q < kvalid ? e0 : 0.f; e1 = q + 1 < kvalid ? e1 : 0.f;
                        f0 = q + 32 < kvalid ? f0 : 0.f; f1 = q + 33 < kvalid ? f1 : 0.f;
                    }
                    l0 += e0 + e1;
                    l1 += f0 + f1;
                    pk[q >> 1] = pack_bf16(e0, e1);
                    pk[16 + (q >> 1)] = pack_bf16(f0, f1);
                }
                l += l0 + l1;
            }
            const bool any_grow = __any_sync(0xffffffffu, grow) && i > 0;
            if (i > 0) {
                // P and O are free once the previous tile's P.V product has completed
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->pv_done), (i - 1) & 1, abort_flag)) && ok;
                tc_fence_after();
            }
            if (any_grow) {                                        // this warp's half of the row's accumulator columns
#pragma unroll 1
                for (uint32_t c = 0; c < 128u; c += 32u) {
                    const uint32_t at = tmem + lane_base + (uint32_t)(warp >> 2) * 128u + c;
                    uint32_t r[32];
                    tmem_ld32(at, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 32; ++q) r[q] = __float_as_uint(__uint_as_float(r[q]) * factor);
                    tmem_st32(at, r);
                }
                tmem_st_wait();
            }
            // swizzled store (row r, 16-byte chunk c -> c ^ (r & 7))
            uint8_t* prow = smem_p + kb * BLOCK_BYTES + row * 128;
#pragma unroll
            for (int g = 0; g < 8; ++g)
                *(uint4*)(prow + ((g ^ (row & 7)) << 4)) = make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
            tc_fence_before();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_bar(&bars->p_full));
        }
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->pv_done), (j1 - j0 - 1) & 1, abort_flag)) && ok;
        tc_fence_after();
        // the row's sum over its four threads
        red[kb * ROWS] = l;
        named_barrier_sync(1 + (quarter & 1), SOFTMAX_WARPS * 16);
        l = (red[0] + red[ROWS]) + (red[2 * ROWS] + red[3 * ROWS]);
        if (ok) {
            const float inv = 1.f / l;
            const bool inside = q0 + row < a.T;
            const int ch0 = (warp >> 2) * 256 + (quarter >> 1) * 128;      // this thread's 128 channels
            __nv_bfloat16* orow = (__nv_bfloat16*)a.o + ((size_t)b * a.T + q0 + row) * a.ld_o + ch0;
#pragma unroll 1
            for (int c = 0; c < 128; c += 32) {
                uint32_t r[32];
                tmem_ld32(tmem + lane_base + (uint32_t)((warp >> 2) * 128 + c), r);
                tmem_ld_wait();
                if (a.splits > 1) {
#pragma unroll
                    for (int q = 0; q < 32; q += 4)
                        *(uint4*)(smem_st + dump_at(row, (ch0 + c + q) >> 2)) = make_uint4(r[q], r[q + 1], r[q + 2], r[q + 3]);
                } else if (inside) {
#pragma unroll
                    for (int q = 0; q < 32; q += 8) {
                        float v[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[q + e]) * inv;
                        *(uint4*)(orow + c + q) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]),
                                                             pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
                    }
                }
            }
        }
    } else if (warp == LOAD_WARP) {
        // ------------------------------------------------------------ loads, in the order of their use: K(0), K(1), V(0), K(2), V(1), ...
        if (lane == 0) {
            const uint32_t qbar = leader_bar(&bars->q_full);
            mbar_arrive_expect_tx_cluster(qbar, Q_BYTES);
            for (int c = 0; c < QK_CHUNKS; ++c)
                tma_load_2d_pair(smem_u32(smem_q + c * BLOCK_BYTES), &tm_q, c * CHUNK, b * a.T + q0, qbar);
            uint32_t st = 0, ph = 0;
            int issued = 0;
            auto load = [&](const CUtensorMap* tm, int x0, int y0, int x1, int y1) -> bool {
                if (!mbar_wait(smem_u32(&bars->empty[st]), ph ^ 1, abort_flag)) return false;
                const uint32_t full = leader_bar(&bars->full[st]);
                mbar_arrive_expect_tx_cluster(full, STAGE_BYTES);
                tma_load_2d_pair(smem_u32(smem_st + st * STAGE_BYTES), tm, x0, y0, full);
                tma_load_2d_pair(smem_u32(smem_st + st * STAGE_BYTES + BOX_BYTES), tm, x1, y1, full);
                ++issued;
                if (++st == STAGES) { st = 0; ph ^= 1; }
                return true;
            };
            auto load_k = [&](int j) {
                const int y = b * a.T + j * BKV + (int)rank * 128;
                for (int c = 0; c < QK_CHUNKS && ok; c += 2) ok = load(&tm_k, c * CHUNK, y, (c + 1) * CHUNK, y);
            };
            auto load_v = [&](int j) {
                const int blocks = (min(BKV, a.T - j * BKV) + 63) >> 6;
                const int x = j * BKV, y = b * CH + (int)rank * 128;
                for (int k = 0; k < blocks && ok; ++k) ok = load(&tm_vt, x + k * 64, y, x + k * 64, y + 256);
            };
            load_k(j0);
            for (int j = j0; j < j1 && ok; ++j) {
                if (j + 1 < j1) load_k(j + 1);
                if (ok) load_v(j);
            }
            // Everything has landed once it has been multiplied.  If a wait gave up anywhere, what is on its way lands before the
            // CTA's memory goes (both CTAs' loads are counted in the pair's first one; the other one lets the limit pass).
            for (int k = 0; k < STAGES && ok; ++k) {
                ok = mbar_wait(smem_u32(&bars->empty[st]), ph ^ 1, abort_flag);
                if (ok && ++st == STAGES) { st = 0; ph ^= 1; }
            }
            if (!ok && rank == 0) {
                cc::land_loads(&bars->q_full, 1, 1);
                cc::land_loads(bars->full, STAGES, issued);
            } else if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < WAIT_LIMIT_CYCLES) {}
            }
        }
    } else if (rank == 0) {
        // ------------------------------------------------------------ MMA issue (the pair's first CTA)
        // The whole warp runs the loop and the tensor instructions are predicated on one elected lane
        // (no branch): warp-uniform code keeps the descriptors in uniform registers, which makes the
        // wait / 4 x MMA / commit sequence of a stage cheaper than the 256 tensor cycles it
        // feeds.  The waits are not voted on (a wait that gave up leaves garbage behind that nobody
        // reads); the abort flag is looked at once per key tile.
        const uint32_t on = elect_one();
        constexpr uint32_t idesc = make_idesc_bf16(128, 256);
        const uint32_t hi = desc_hi(1024, 2);
        const uint32_t peer = crank | 1u;
        uint32_t st = 0, ph = 0;
        auto wait_on = [&](uint64_t* bar, uint32_t parity) {
            const uint32_t p = smem_u32(bar);
            if (!mbar_try_wait(p, parity)) (void)mbar_wait(p, parity, abort_flag);
            tc_fence_after();
        };
        auto commit = [&](uint64_t* bar) { umma2_commit_pair_on(smem_u32(bar), map_to_cta(smem_u32(bar), peer), on); };
        // box i of the stage times operand a_i into accumulator d_i
        auto stage_mmas = [&](uint32_t d0, uint32_t a0, uint32_t d1, uint32_t a1, uint32_t acc0, uint32_t acc1) {
            wait_on(&bars->full[st], ph);
            const uint32_t b_lo = desc_lo(smem_u32(smem_st + st * STAGE_BYTES)), b_lo1 = b_lo + (BOX_BYTES >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma2_bf16_split_on(d0, a0 + k * 2, hi, b_lo + k * 2, hi, idesc, (k == 0) ? acc0 : 1u, on);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma2_bf16_split_on(d1, a1 + k * 2, hi, b_lo1 + k * 2, hi, idesc, (k == 0) ? acc1 : 1u, on);
            commit(&bars->empty[st]);
            __syncwarp();
            if (++st == STAGES) { st = 0; ph ^= 1; }
        };
        const uint32_t q_lo = desc_lo(smem_u32(smem_q)), p_lo = desc_lo(smem_u32(smem_p));
        auto issue_qk = [&](int i) {
            const uint32_t d = tmem_s + (uint32_t)(i & 1) * 128u;
            wait_on(&bars->s_free[i & 1], ((i >> 1) & 1) ^ 1);
            for (int c = 0; c < QK_CHUNKS; c += 2) {
                const uint32_t q = q_lo + (uint32_t)(c * (BLOCK_BYTES >> 4));
                stage_mmas(d, q, d, q + (BLOCK_BYTES >> 4), c != 0 ? 1u : 0u, 1u);
            }
            commit(&bars->s_full[i & 1]);
            __syncwarp();
        };
        auto issue_pv = [&](int i, int blocks) {
            wait_on(&bars->p_full, i & 1);
            for (int k = 0; k < blocks; ++k) {
                const uint32_t p = p_lo + (uint32_t)(k * (BLOCK_BYTES >> 4)), acc = (i | k) != 0 ? 1u : 0u;
                stage_mmas(tmem, p, tmem + 128u, p, acc, acc);
            }
            commit(&bars->pv_done);
            __syncwarp();
        };
        wait_on(&bars->q_full, 0);
        issue_qk(0);
        for (int j = j0; j < j1; ++j) {
            if (*abort_flag) break;
            if (j + 1 < j1) issue_qk(j + 1 - j0);
            issue_pv(j - j0, (min(BKV, a.T - j * BKV) + 63) >> 6);
        }
        if (*abort_flag) {                                   // nobody else waits for the products under way
            commit(&bars->drained);
            __syncwarp();
            (void)cc::wait_cluster(smem_u32(&bars->drained), 0, abort_flag);
            __syncwarp();
        }
    }

    tc_fence_before();
    __syncthreads();
    if (a.splits > 1) {
        // each CTA finishes its share of the 64 rows x 64 pieces of eight channels that the cluster's CTAs of its rank hold
        float2* ml = (float2*)s_red;                                  // (every sum above has been read)
        if (warp < 4 && kb == 0) ml[row] = make_float2(m_ref, l);
        cluster_sync_all();
        if (warp < SOFTMAX_WARPS) {
            constexpr int ITEMS = ROWS * CH / 8;
            const uint32_t base = smem_u32(smem_st), ml_base = smem_u32(ml);
            for (int it = ITEMS * split / a.splits + tid; it < ITEMS * (split + 1) / a.splits; it += SOFTMAX_WARPS * 32) {
                const int r = it / (CH / 8), piece = (it % (CH / 8)) * 2;
                float2 w[kMaxSplits];
                float4 lo[kMaxSplits], hi4[kMaxSplits];
#pragma unroll
                for (int s = 0; s < kMaxSplits; ++s) {
                    if (s < a.splits) {
                        const uint32_t cta = 2u * (uint32_t)s + rank;
                        w[s] = ld_cluster_f2(map_to_cta(ml_base + (uint32_t)r * 8u, cta));
                        lo[s] = ld_cluster_f4(map_to_cta(base + dump_at(r, piece), cta));
                        hi4[s] = ld_cluster_f4(map_to_cta(base + dump_at(r, piece + 1), cta));
                    }
                }
                float m = w[0].x;
#pragma unroll
                for (int s = 1; s < kMaxSplits; ++s) if (s < a.splits) m = fmaxf(m, w[s].x);
                float sum = 0.f, v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int s = 0; s < kMaxSplits; ++s) {
                    if (s < a.splits) {
                        const float f = ex2(w[s].x - m);
                        sum = fmaf(f, w[s].y, sum);
                        v[0] = fmaf(f, lo[s].x, v[0]); v[1] = fmaf(f, lo[s].y, v[1]); v[2] = fmaf(f, lo[s].z, v[2]); v[3] = fmaf(f, lo[s].w, v[3]);
                        v[4] = fmaf(f, hi4[s].x, v[4]); v[5] = fmaf(f, hi4[s].y, v[5]); v[6] = fmaf(f, hi4[s].z, v[6]); v[7] = fmaf(f, hi4[s].w, v[7]);
                    }
                }
                if (q0 + r < a.T) {
                    const float inv = 1.f / sum;
                    *(uint4*)((__nv_bfloat16*)a.o + ((size_t)b * a.T + q0 + r) * a.ld_o + piece * 4) =
                        make_uint4(pack_bf16(v[0] * inv, v[1] * inv), pack_bf16(v[2] * inv, v[3] * inv),
                                   pack_bf16(v[4] * inv, v[5] * inv), pack_bf16(v[6] * inv, v[7] * inv));
                }
            }
        }
    }
    cluster_sync_all();                                               // nobody leaves while others may still touch its memory
    if (tid == 0 && bars->abort_flag && status) {
        if (atomicCAS(status, 0u, kStatusAttnTimeout) == 0u) {
            status[1] = blockIdx.x;
            status[2] = 0;
        }
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc2(tmem, 512);
    }
}

// Up to 128 tokens: one tile of everything, so the kernel is a chain of latencies (loads, scores, softmax, P V, output) without
// a loop, and a cluster's barriers would only lengthen it (with the transpose, us: 64 tokens 12.3, on a pair 16.6, on the kernel
// before these 13.9; 128 tokens 12.4, 15.4, 14.4).  A CTA takes all the queries and 128 channels of the output, and computes the
// scores for itself.
constexpr int SMALL = 128, SMALL_STAGES = 5, SMALL_STAGE_BYTES = 2 * SMALL * CHUNK * 2;      // Q chunk + K chunk
constexpr int SMALL_V_BYTES = 2 * 128 * CHUNK * 2;           // 128 channels x 2 x 64 keys
constexpr int SMALL_SMEM = SMALL_STAGES * SMALL_STAGE_BYTES + SMALL_V_BYTES + 4 * SMALL * 4 + 256 + 1024;
struct SmallBars {
    uint64_t qk_full[SMALL_STAGES], qk_empty[SMALL_STAGES], v_full, s_full, p_full, o_full;
    uint32_t tmem_base, abort_flag;
};
static_assert(sizeof(SmallBars) <= 256 && SMALL_SMEM <= 232448 && 2 * SMALL * 128 <= SMALL_STAGE_BYTES, "shared memory of one CTA; P lies over the first stage");

__global__ void __launch_bounds__(NUM_THREADS, 1)
attn_small_kernel(const AttnTcParams a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                  const __grid_constant__ CUtensorMap tm_vt, unsigned int* status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* smem_v = smem + SMALL_STAGES * SMALL_STAGE_BYTES;
    float* s_red = (float*)(smem_v + SMALL_V_BYTES);         // [2 x maximum, 2 x sum][SMALL]
    SmallBars* bars = (SmallBars*)(s_red + 4 * SMALL);
    volatile uint32_t* abort_flag = &bars->abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ch0 = (int)(blockIdx.x % (CH / 128)) * 128, b = (int)blockIdx.x / (CH / 128);
    const int blocks = (a.T + 63) >> 6;                      // 64-key blocks that exist
    if (tid == 0) {
        for (int i = 0; i < SMALL_STAGES; ++i) { mbar_init(smem_u32(&bars->qk_full[i]), 1); mbar_init(smem_u32(&bars->qk_empty[i]), 1); }
        mbar_init(smem_u32(&bars->v_full), 1);
        mbar_init(smem_u32(&bars->s_full), 1);
        mbar_init(smem_u32(&bars->p_full), SOFTMAX_WARPS);
        mbar_init(smem_u32(&bars->o_full), 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
    }
    if (warp == MMA_WARP) tmem_alloc(smem_u32(&bars->tmem_base), 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base, tmem_o = tmem + 128;
    griddep_launch();
    if (warp != MMA_WARP) griddep_wait();
    if (warp < SOFTMAX_WARPS) {
        // ------------------------------------------------ two threads per query row, 64 keys each
        const int row = (warp & 3) * 32 + lane, kb = warp >> 2;
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->s_full), 0, abort_flag));
        tc_fence_after();
        uint32_t r0[32], r1[32];
        tmem_ld32(tmem + lanes + (uint32_t)kb * 64u, r0);
        tmem_ld32(tmem + lanes + (uint32_t)kb * 64u + 32u, r1);
        tmem_ld_wait();
        const int kvalid = min(max(a.T - kb * 64, 0), 64);
        float m = -INFINITY;
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            if (q < kvalid) m = fmaxf(m, __uint_as_float(r0[q]) * a.scale_log2);
            if (q + 32 < kvalid) m = fmaxf(m, __uint_as_float(r1[q]) * a.scale_log2);
        }
        s_red[kb * SMALL + row] = m;
        named_barrier_sync(1, SOFTMAX_WARPS * 32);
        m = fmaxf(s_red[row], s_red[SMALL + row]);
        float l = 0.f;
        uint32_t pk[32];
#pragma unroll
        for (int q = 0; q < 32; q += 2) {
            float e[4] = {ex2(fmaf(__uint_as_float(r0[q]), a.scale_log2, -m)), ex2(fmaf(__uint_as_float(r0[q + 1]), a.scale_log2, -m)),
                          ex2(fmaf(__uint_as_float(r1[q]), a.scale_log2, -m)), ex2(fmaf(__uint_as_float(r1[q + 1]), a.scale_log2, -m))};
            e[0] = q < kvalid ? e[0] : 0.f; e[1] = q + 1 < kvalid ? e[1] : 0.f;
            e[2] = q + 32 < kvalid ? e[2] : 0.f; e[3] = q + 33 < kvalid ? e[3] : 0.f;
            l += (e[0] + e[1]) + (e[2] + e[3]);
            pk[q >> 1] = pack_bf16(e[0], e[1]);
            pk[16 + (q >> 1)] = pack_bf16(e[2], e[3]);
        }
        uint8_t* prow = smem + kb * (SMALL * 128) + row * 128;       // (every score is there: the stages are free)
#pragma unroll
        for (int g = 0; g < 8; ++g)
            *(uint4*)(prow + ((g ^ (row & 7)) << 4)) = make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
        tc_fence_before();
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->p_full));
        s_red[(2 + kb) * SMALL + row] = l;
        named_barrier_sync(1, SOFTMAX_WARPS * 32);
        const float inv = 1.f / (s_red[2 * SMALL + row] + s_red[3 * SMALL + row]);
        ok = ok && __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->o_full), 0, abort_flag));
        tc_fence_after();
        if (ok) {
            tmem_ld32(tmem_o + lanes + (uint32_t)kb * 64u, r0);
            tmem_ld32(tmem_o + lanes + (uint32_t)kb * 64u + 32u, r1);
            tmem_ld_wait();
            if (row < a.T) {
                __nv_bfloat16* o = (__nv_bfloat16*)a.o + ((size_t)b * a.T + row) * a.ld_o + ch0 + kb * 64;
#pragma unroll
                for (int q = 0; q < 64; q += 8) {
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(q < 32 ? r0[(q + e) & 31] : r1[(q + e) & 31]) * inv;
                    *(uint4*)(o + q) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
                }
            }
        }
    } else if (warp == LOAD_WARP) {
        if (lane == 0) {
            for (int c = 0; c < QK_CHUNKS; ++c) {
                const int st = c % SMALL_STAGES;
                if (c >= SMALL_STAGES && !mbar_wait(smem_u32(&bars->qk_empty[st]), 0, abort_flag)) break;
                const uint32_t full = smem_u32(&bars->qk_full[st]);
                uint8_t* dst = smem + st * SMALL_STAGE_BYTES;
                mbar_arrive_expect_tx(full, SMALL_STAGE_BYTES);
                tma_load_2d(smem_u32(dst), &tm_q, c * CHUNK, b * a.T, full);
                tma_load_2d(smem_u32(dst + SMALL * CHUNK * 2), &tm_k, c * CHUNK, b * a.T, full);
                if (c == SMALL_STAGES - 1) {
                    const uint32_t vf = smem_u32(&bars->v_full);
                    mbar_arrive_expect_tx(vf, (uint32_t)blocks * (SMALL_V_BYTES / 2));
                    for (int k = 0; k < blocks; ++k) tma_load_2d(smem_u32(smem_v + k * (SMALL_V_BYTES / 2)), &tm_vt, k * 64, b * CH + ch0, vf);
                }
            }
            // (all loads have landed when the product is complete; if a wait gave up, before the CTA's memory goes)
            if (!mbar_wait(smem_u32(&bars->o_full), 0, abort_flag)) {
                for (int i = 0; i < SMALL_STAGES; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(smem_u32(&bars->qk_full[i]), 0) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
                }
                for (int i = 0; i < QK_CHUNKS - SMALL_STAGES; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(smem_u32(&bars->qk_full[i]), 1) && clock64() - t0 < WAIT_LIMIT_CYCLES / 16) {}
                }
                const long long t0 = clock64();
                while (!mbar_try_wait(smem_u32(&bars->v_full), 0) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
            }
        }
    } else {
        const uint32_t on = elect_one();
        constexpr uint32_t idesc = make_idesc_bf16(128, 128);
        const uint32_t hi = desc_hi(1024, 2);
        auto wait_on = [&](uint64_t* bar, uint32_t parity) {
            (void)mbar_wait(smem_u32(bar), parity, abort_flag);
            tc_fence_after();
        };
        for (int c = 0; c < QK_CHUNKS; ++c) {
            const int st = c % SMALL_STAGES;
            wait_on(&bars->qk_full[st], c >= SMALL_STAGES ? 1u : 0u);
            const uint32_t qa = desc_lo(smem_u32(smem + st * SMALL_STAGE_BYTES)), ka = qa + ((SMALL * CHUNK * 2) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_bf16_split_on(tmem, qa + k * 2, hi, ka + k * 2, hi, idesc, (c | k) != 0 ? 1u : 0u, on);
            if (c + SMALL_STAGES < QK_CHUNKS) umma_commit_on(smem_u32(&bars->qk_empty[st]), on);
            __syncwarp();
        }
        umma_commit_on(smem_u32(&bars->s_full), on);
        __syncwarp();
        wait_on(&bars->v_full, 0);
        wait_on(&bars->p_full, 0);
        for (int k = 0; k < blocks; ++k) {
            const uint32_t pa = desc_lo(smem_u32(smem + k * (SMALL * 128))), va = desc_lo(smem_u32(smem_v + k * (SMALL_V_BYTES / 2)));
#pragma unroll
            for (int i = 0; i < 4; ++i) umma_bf16_split_on(tmem_o, pa + i * 2, hi, va + i * 2, hi, idesc, (k | i) != 0 ? 1u : 0u, on);
        }
        umma_commit_on(smem_u32(&bars->o_full), on);
        __syncwarp();
        if (*abort_flag) (void)cc::wait_cluster(smem_u32(&bars->o_full), 0, abort_flag);     // (the others no longer wait for the products under way)
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && bars->abort_flag && status) {
        if (atomicCAS(status, 0u, kStatusAttnTimeout) == 0u) {
            status[1] = blockIdx.x;
            status[2] = 0;
        }
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem, 256);
    }
}

// v [B][T][ld] -> vt [B][C][Tp] (tokens contiguous, zero beyond T)
__global__ void transpose_v_kernel(const __nv_bfloat16* v, __nv_bfloat16* vt, int T, int Tp, int C, int ld) {
    __shared__ __nv_bfloat16 tile[32][33];
    griddep_launch();
    griddep_wait();
    const int b = blockIdx.z;
    const int t0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int t = t0 + i, c = c0 + threadIdx.x;
        tile[i][threadIdx.x] = (t < T) ? v[((size_t)b * T + t) * ld + c] : __float2bfloat16(0.f);
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int c = c0 + i, t = t0 + threadIdx.x;
        if (t < Tp) vt[((size_t)b * C + c) * Tp + t] = tile[threadIdx.x][i];
    }
}

bool encode_2d(CUtensorMap* tm, const void* base, uint64_t cols, uint64_t rows, uint64_t row_stride_bytes, uint32_t box_cols,
               uint32_t box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {row_stride_bytes};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int padded_tokens(int T) { return (T + 63) / 64 * 64; }

// clusters of 2 * splits CTAs that the current device holds at once (0: none), asked once per device
int max_clusters(int splits) {
    static std::mutex mu;
    static int known[cc::kMaxDevices][kMaxSplits] = {};      // 0: not asked, else the answer + 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= cc::kMaxDevices || cc::set_smem_limit<attn_tc_kernel>(SMEM_TOTAL) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    std::lock_guard<std::mutex> lock(mu);
    int& k = known[dev][splits - 1];
    if (k == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2u * (unsigned)splits);
        cfg.blockDim = dim3(NUM_THREADS);
        cfg.dynamicSmemBytes = SMEM_TOTAL;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2u * (unsigned)splits; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, (const void*)attn_tc_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        k = n + 1;
    }
    return k - 1;
}

// Pairs that share a query tile's keys: the fewest rounds of clusters x (key tiles of a pair + what a cluster costs besides, in
// tiles: its fill, and the exchange where the keys are divided).  0: the device cannot hold a pair.
// Measured with 1 / 2 / 3 / 4 pairs, us, the same call again and again (what the rule takes in brackets): 400 tokens [18.5] / 20.2, 1024
// 22.6 / [22.5] / 22.6 / 22.6, 1537 30.0 / 27.7 / 25.8 / [25.7], 1791 32.8 / 28.7 / 28.7 / [26.7], 1961 34.9 / [28.7] / 28.7 / 43.1, 2200 36.9 / 30.8 /
// [30.0] / 48.3, 3000 43.1 / [34.9] / 53.3 / 50.7, 3600 53.0 / [41.0] / 61.4 / 57.5, 5400 [71.7] / 86.1 / 77.9 / 96.5, two times 5400 137 / [132] / 147 /
// 187, eight times [406] / 494 / 586 / 706, 14400 369 / [384] / 405 / 409, two times 746 / [738] / 784 / 876, four times 1024 32.3 / [34.8] / 54.3 / 59.6.
int choose_splits(int B, int T, bool no_clusters) {
    const long long q_tiles = (long long)((T + BQ - 1) / BQ) * std::max(B, 1);
    const int ntiles = (T + BKV - 1) / BKV;
    int best = 0;
    double best_cost = 0.0;
    for (int s = 1; s <= (no_clusters ? 1 : kMaxSplits) && s <= ntiles; ++s) {
        const int n = max_clusters(s);
        if (n < 1) continue;
        const double cost = (double)((q_tiles + n - 1) / n) * ((ntiles + s - 1) / s + (s == 1 ? 1.0 : s == 2 ? 2.5 : 4.0));
        if (best == 0 || cost < best_cost) { best = s; best_cost = cost; }
    }
    return best;
}

}  // namespace

bool attn_tc_supported(const AttnArgs& a) {
    return a.dtype == VD_BF16 && a.C == CH && a.ld_qkv % 8 == 0 && a.ld_o % 8 == 0 && a.T >= 1;
}
bool attn_tc_available() { return max_clusters(1) >= 1; }

size_t attn_tc_scratch_bytes(int B, int T, int C) { return (size_t)B * C * padded_tokens(T) * 2; }

cudaError_t attn_tc_prepare(const AttnArgs& a, AttnTcPlan* plan) {
    plan->valid = 0;
    if (!a.vt) return cudaErrorInvalidValue;
    if (((uintptr_t)a.q | (uintptr_t)a.k | (uintptr_t)a.vt) & 15) return cudaErrorMisalignedAddress;
    const int Tp = padded_tokens(a.T);
    const uint64_t rows = (uint64_t)a.B * a.T;
    const bool small = a.T <= SMALL;
    if (!encode_2d((CUtensorMap*)plan->tq, a.q, a.C, rows, (uint64_t)a.ld_qkv * 2, CHUNK, small ? SMALL : ROWS)) return cudaErrorInvalidValue;
    if (!encode_2d((CUtensorMap*)plan->tk, a.k, a.C, rows, (uint64_t)a.ld_qkv * 2, CHUNK, 128)) return cudaErrorInvalidValue;
    if (!encode_2d((CUtensorMap*)plan->tv, a.vt, Tp, (uint64_t)a.B * a.C, (uint64_t)Tp * 2, CHUNK, 128)) return cudaErrorInvalidValue;
    plan->splits = small ? 0 : choose_splits(a.B, a.T, a.no_clusters != 0);
    if (!small && plan->splits < 1) return cudaErrorInvalidConfiguration;
    plan->q = a.q; plan->k = a.k; plan->vt = a.vt;
    plan->batch = a.B; plan->tokens = a.T;
    plan->valid = 1;
    return cudaSuccess;
}

cudaError_t launch_attn_tc(const AttnArgs& a, const AttnTcPlan* plan, unsigned int* status, cudaStream_t s) {
    if (!a.vt) return cudaErrorInvalidValue;
    if (((uintptr_t)a.q | (uintptr_t)a.k | (uintptr_t)a.v | (uintptr_t)a.o | (uintptr_t)a.vt) & 15) return cudaErrorMisalignedAddress;
    const int Tp = padded_tokens(a.T);
    {
        dim3 grid(Tp / 32, a.C / 32, a.B), block(32, 8);
        cudaError_t e = launch_pdl(transpose_v_kernel, grid, block, 0, s, (const __nv_bfloat16*)a.v, (__nv_bfloat16*)a.vt, a.T, Tp, a.C, a.ld_qkv);
        if (e != cudaSuccess) return e;
    }
    // The maps of a decoder's fixed workspace tensors are built once (attn_tc_prepare, for the largest batch: rows
    // beyond the batch in use are never addressed); a call on other tensors encodes its own.
    AttnTcPlan local;
    if (!(plan && plan->valid && plan->q == a.q && plan->k == a.k && plan->vt == a.vt && plan->tokens == a.T && a.B <= plan->batch)) {
        cudaError_t e = attn_tc_prepare(a, &local);
        if (e != cudaSuccess) return e;
        plan = &local;
    }
    const CUtensorMap &tq = *(const CUtensorMap*)plan->tq, &tk = *(const CUtensorMap*)plan->tk, &tv = *(const CUtensorMap*)plan->tv;
    AttnTcParams p{a.o, a.B, a.T, a.ld_o, plan->splits, a.scale * 1.4426950408889634f};
    if (plan->splits == 0) {
        const cudaError_t e = cc::set_smem_limit<attn_small_kernel>(SMALL_SMEM);
        if (e != cudaSuccess) return e;
        return launch_pdl(attn_small_kernel, dim3((unsigned)(CH / 128) * (unsigned)a.B), dim3(NUM_THREADS), SMALL_SMEM, s, p, tq, tk, tv, status);
    }
    const int cluster = 2 * plan->splits;
    const long long ctas = (long long)((a.T + BQ - 1) / BQ) * cluster * a.B;
    return cc::launch_clusters<attn_tc_kernel>({ctas, NUM_THREADS, SMEM_TOTAL, SMEM_TOTAL, cluster}, s, p, tq, tk, tv, status);
}

}  // namespace vd
