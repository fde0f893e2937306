// Single-precision convolution (3x3, 1x1, upsampling 3x3) as a register-tiled implicit GEMM on the FP32 pipes, with the
// same fusion as the tensor-core kernels: GroupNorm + SiLU in the prologue, bias and residual in the epilogue, and
// the statistics of the next GroupNorm as records (conv_cluster.cuh).
//
//   * A CTA of 256 threads computes a tile of TH x 8 pixels x 32 output channels over its share of the input channels;
//     a thread holds 8 pixels of a row x 4 channels.  Per input channel and kernel row it reads 10 pixels and 3 x 4
//     weights (6 shared loads of 16 bytes, none conflicting) for 96 multiply-adds, issued as fma.rn.f32x2: the FMA pipes
//     are the bound.  Products and sums are IEEE fp32, as in the direct kernel (kernels_simt.cu), in another order.
//   * K is divided twice where the image is small: KT thread groups of the CTA take every KT-th channel of a chunk, and
//     a cluster of up to 8 CTAs takes a share of the chunks each.  Partials meet in shared memory.
//   * Weights (fp32 [tap][Cin][Cout]) come by bulk tensor loads, as many chunks ahead as shared memory holds, and do not
//     wait for the kernel before (programmatic dependent launch).
//   * A nearest-2x upsampling 3x3 is four 2x2 convolutions of the source with weights summed in advance (fp32), one per
//     output parity: 16 instead of 36 products per source pixel.
// Measured on one B200 (profiled launches, direct kernel -> this one): 512->512 at 8x8 613 -> 31 us, at 16x16 604 -> 48;
// 32->32 on four 256x256 frames 414 -> 142; frame head 32->3 on a 64x64 frame 29 -> 12, on four 256x256 frames (32-pixel tiles)
// 83 -> 59.  Whole decodes, with the statistics as records: tiny layout 64x64 652 -> 127 us, full-width layout 64x64
// 16.5 -> 1.25 ms.
#include <string.h>

#include <algorithm>

#include "conv_cluster.cuh"

namespace vd {

namespace {

using namespace cc;
using namespace tc;

constexpr int kThreads = 256, kChunk = 16;                   // threads, input channels per chunk
constexpr int kMaxW = 8;                                     // weight stages

enum { K3X3 = 0, K1X1 = 1, KPHASE = 2 };

__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long both(float x) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
    return d;
}
__device__ __forceinline__ float2 halves(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, int x, int y, int z, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}

__device__ __forceinline__ unsigned long long pair(float x, float y) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
struct FBars {
    uint64_t w_full[kMaxW];
    uint64_t rx_full;
    uint32_t abort_flag, unused;
    int issued;                                              // weight loads
};

// Geometry of a build: a tile of TH x TW pixels (a thread has eight pixels of a row).  BN = 4: the frame head (at most four
// output channels; its weights are read with plain loads).
template <int TH, int BN, int KIND, int TW = 8> struct FCfg {
    static constexpr int KH = KIND == K3X3 ? 3 : (KIND == K1X1 ? 1 : 2), TAPS = KH * KH;
    static constexpr int RH = TH + KH - 1, RW = TW + KH - 1;            // rows and columns of the input tile
    static constexpr int ROW = TW + 4;                                   // floats per tile row (16-byte rows; KH - 1 of the four extra ones used)
    static constexpr int CS = (RH * ROW + 7) / 8 * 8 + 4;                // floats per channel: four channels of a pixel on distinct banks
    static constexpr int NG = TW / 8, KT = kThreads / (TH * NG * (BN / 4));             // thread groups along K
    static constexpr int IN_FLOATS = kChunk * CS;
    static constexpr int W_FLOATS = TAPS * kChunk * BN;
    static constexpr int RX_FLOATS = TH * TW * BN;                       // one partial of the tile
    static constexpr int PART_FLOATS = KT / 2 * RX_FLOATS;               // partials of half the K groups at a time
    static_assert(KT >= 2 && kThreads % (TH * NG * (BN / 4)) == 0 && CS % 4 == 0, "thread layout");
};
constexpr int kMaxSlice = 512, kMaxSplits = kF32MaxSplits;   // input channels of one CTA; CTAs of a cluster
constexpr int kFTail = 2 * kMaxSlice * 4 + 128;              // scale / shift of the slice, barriers
static_assert(sizeof(FBars) <= 128, "barrier block");

// A partial lies in memory as rows (pixels) of BN floats whose 16-byte pieces are permuted by the row, so that neither the
// threads that write it (eight tile rows side by side) nor those that read it (eight pixels of a row) meet on a bank.
// The frame head's rows are one piece long: there the pixels of a group of eight are permuted (displacement of row R).
template <int BN, int TW> __device__ __forceinline__ int piece(int R) { return BN < 32 ? ((R ^ (R / TW)) & 7) - (R & 7) : (R ^ (R >> 3)) & 7; }

template <int TH, int BN, int KIND, int TW>
__global__ void __launch_bounds__(kThreads, 2)
conv_f32_kernel(const ConvArgs a, const int S, const int n_w, const int ops_floats, const __grid_constant__ CUtensorMap tm_w, unsigned int* status) {
    using C = FCfg<TH, BN, KIND, TW>;
    constexpr bool HEAD = BN < 32;
    constexpr int KH = C::KH, CS = C::CS, KT = C::KT, ROW = C::ROW;
    static_assert(TW == 8 || HEAD, "wide tiles");
    extern __shared__ uint8_t smem_raw[];
    float* s_in = (float*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);           // two input chunks
    float* s_w = s_in + (2 * C::IN_FLOATS + 31) / 32 * 32;                           // n_w weight stages (head: the whole slice)
    float* rx = s_in + ops_floats;                                                   // partials of this CTA's rows
    float* part = s_in;                                                              // this CTA's partials, once every thread is done with its operands
    float* s_scale = s_in + ops_floats + (S > 1 ? C::RX_FLOATS : 0);
    float* s_shift = s_scale + kMaxSlice;
    FBars* bars = (FBars*)(s_shift + kMaxSlice);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, lane = tid & 31;
    const int rank = S > 1 ? (int)cluster_ctarank() : 0;
    const int H = KIND == KPHASE ? a.Hs : a.H, W = KIND == KPHASE ? a.Ws : a.W;      // the tile grid is that of the source
    const int tiles_x = (W + TW - 1) / TW, tiles = tiles_x * ((H + TH - 1) / TH);
    const int nblk = HEAD ? 1 : a.Cout / BN;
    int item = (int)blockIdx.x / S;
    const int n0 = (item % nblk) * BN;
    item /= nblk;
    const int par = KIND == KPHASE ? (item & 3) : 0;
    if (KIND == KPHASE) item >>= 2;
    const int tile = item % tiles, frame = item / tiles;
    const int ty = (tile / tiles_x) * TH, tx = (tile % tiles_x) * TW;
    const int oy0 = KIND == K3X3 ? -1 : (KIND == KPHASE ? (par >> 1) - 1 : 0), ox0 = KIND == K3X3 ? -1 : (KIND == KPHASE ? (par & 1) - 1 : 0);
    const int chunks = (a.Cin + kChunk - 1) / kChunk;
    const int k0 = rank * chunks / S, units = (rank + 1) * chunks / S - k0;
    const int c_first = k0 * kChunk, nch = min(a.Cin - c_first, units * kChunk);

    auto load_weights = [&](int u) {                         // chunk u of the slice into its stage
        const uint32_t full = smem_u32(&bars->w_full[u % n_w]);
        mbar_arrive_expect_tx(full, C::W_FLOATS * 4);
        tma_load_3d(smem_u32(s_w + (u % n_w) * C::W_FLOATS), &tm_w, n0, c_first + u * kChunk, par * C::TAPS, full);
    };
    if (tid == 0) {
        for (int i = 0; i < kMaxW; ++i) mbar_init(smem_u32(&bars->w_full[i]), 1);
        mbar_init(smem_u32(&bars->rx_full), 1);
        bars->abort_flag = 0;
        bars->issued = HEAD ? 0 : min(units, n_w);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(smem_u32(&bars->rx_full), C::RX_FLOATS * 4);           // this CTA's rows from all S * KT partials
        if (!HEAD)
            for (int u = 0; u < min(units, n_w); ++u) load_weights(u);
    }
    if (HEAD) {                                              // [chunk][tap][16][4], zero beyond Cout and Cin
        for (int i = tid; i < units * C::TAPS * kChunk; i += kThreads) {
            const int u = i / (C::TAPS * kChunk), tap = (i / kChunk) % C::TAPS, c = c_first + u * kChunk + i % kChunk;
            float w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = (q < a.Cout && c < a.Cin) ? __ldg((const float*)a.w + ((size_t)tap * a.Cin + c) * a.Cout + q) : 0.f;
            *(float4*)(s_w + i * 4) = make_float4(w[0], w[1], w[2], w[3]);
        }
    }
    __syncthreads();
    if (S > 1) cluster_arrive();                             // (waited for before anything is sent to another CTA)
    griddep_launch();

    // ---- input: entry e of a thread is (pixel, four channels) of the tile
    constexpr int NE = (C::RH * C::RW * (kChunk / 4) + kThreads - 1) / kThreads;
    const bool prologue = a.scale != nullptr || a.in_rec != nullptr, silu = a.silu != 0, round = a.bf16_operands != 0;
    float4 raw[NE];
    uint32_t vm = 0u;                                        // entries inside the image
    unsigned int src[NE];                                    // in pieces of four channels
    const float4* const image = (const float4*)((const float*)a.x + (size_t)frame * H * W * a.Cin + c_first);
    const int quad = tid & 3;
#pragma unroll
    for (int e = 0; e < NE; ++e) {
        const int pix = (e * kThreads + tid) >> 2, py = pix / C::RW, px = pix - py * C::RW;
        const int y = ty + oy0 + py, x = tx + ox0 + px;
        const bool v = py < C::RH && y >= 0 && y < H && x >= 0 && x < W;
        vm |= (v ? 1u : 0u) << e;
        src[e] = v ? (unsigned int)(y * W + x) * (unsigned int)(a.Cin >> 2) + quad : 0u;
    }
    auto fetch = [&](int u) {
        const bool on = u * kChunk + quad * 4 < nch;         // (Cin is a multiple of 4)
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            raw[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (on && (vm >> e & 1u)) raw[e] = __ldcg(image + src[e] + u * (kChunk / 4));
        }
    };
    InputStats st;
    if (a.in_rec) st.prepare(a, frame, c_first, nch, tid >> 5, lane, s_scale, s_shift);
    if (tid < 32) touch_params(a, &bars->unused);
    griddep_wait();                                          // everything above is arithmetic, weights and parameters
    if (a.in_rec) st.load(a, lane);
    fetch(0);
    if (prologue) {
        if (a.in_rec) st.finish(a, nch, lane, 1.f, s_scale, s_shift);
        else
            for (int c = tid; c < nch; c += kThreads) {
                s_scale[c] = __ldcg(a.scale + (size_t)frame * a.Cin + c_first + c);
                s_shift[c] = __ldcg(a.shift + (size_t)frame * a.Cin + c_first + c);
            }
        __syncthreads();
    }

    // thread = (K group, 4 channels, tile row); a warp holds 8 rows x 4 channel columns (head: 16 rows x 2 K groups)
    const int ng = HEAD && TW > 8 ? tid / TH % C::NG : 0;    // eight-pixel group of the row
    const int row = HEAD ? tid % TH : (TH == 8 ? tid & 7 : (tid & 7) + ((tid >> 6) & 1) * 8);
    const int cg = HEAD ? 0 : (tid >> 3) & 7;
    const int kt = HEAD ? tid / (TH * C::NG) : tid / (TH * (BN / 4));
    unsigned long long acc[8][2];
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[p][0] = acc[p][1] = 0ull;

#pragma unroll 1
    for (int u = 0; u < units; ++u) {
        float* buf = s_in + (u & 1) * C::IN_FLOATS;
        {
            float4 sc = make_float4(1.f, 1.f, 1.f, 1.f), sf = make_float4(0.f, 0.f, 0.f, 0.f);
            const int c = u * kChunk + quad * 4;
            if (prologue && c < nch) { sc = *(const float4*)(s_scale + c); sf = *(const float4*)(s_shift + c); }
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                const int pix = (e * kThreads + tid) >> 2, py = pix / C::RW, px = pix - py * C::RW;
                if (py >= C::RH) break;
                float v[4] = {raw[e].x, raw[e].y, raw[e].z, raw[e].w};
                if (vm >> e & 1u) {                          // outside the image the transformed tensor is zero
                    const float s4[4] = {sc.x, sc.y, sc.z, sc.w}, f4[4] = {sf.x, sf.y, sf.z, sf.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (prologue) v[q] = fmaf(v[q], s4[q], f4[q]);
                        if (silu) v[q] = v[q] / (1.0f + expf(-v[q]));
                        if (round) v[q] = __bfloat162float(__float2bfloat16_rn(v[q]));
                    }
                }
                float* d = buf + quad * 4 * CS + py * ROW + px;
#pragma unroll
                for (int q = 0; q < 4; ++q) d[q * CS] = v[q];
            }
        }
        if (u + 1 < units) fetch(u + 1);
        __syncthreads();                                     // chunk u is complete; every thread is done with chunk u - 1
        if (!HEAD) {
            if (tid == 0 && u > 0 && u - 1 + n_w < units && !*abort_flag) {
                bars->issued = u + n_w;
                load_weights(u - 1 + n_w);
            }
            (void)mbar_wait(smem_u32(&bars->w_full[u % n_w]), (u / n_w) & 1, abort_flag);
        }
        const float* ip = buf + row * ROW + ng * 8;
        const float* wp = s_w + (HEAD ? u : u % n_w) * C::W_FLOATS + cg * 4;
        const int cmax = min(kChunk, nch - u * kChunk);
#pragma unroll 1
        for (int c = kt; c < cmax; c += KT) {
#pragma unroll
            for (int ky = 0; ky < KH; ++ky) {
                float p[8 + KH];
                const float* q = ip + c * CS + ky * ROW;
                *(float4*)&p[0] = *(const float4*)q;
                *(float4*)&p[4] = *(const float4*)(q + 4);
                if (KH == 3) { const float2 t = *(const float2*)(q + 8); p[8] = t.x; p[9] = t.y; }
                if (KH == 2) p[8] = q[8];
                unsigned long long d[7 + KH];
#pragma unroll
                for (int i = 0; i < 7 + KH; ++i) d[i] = both(p[i]);
#pragma unroll
                for (int kx = 0; kx < KH; ++kx) {
                    const ulonglong2 w = *(const ulonglong2*)(wp + ((ky * KH + kx) * kChunk + c) * BN);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        fma2(acc[i][0], d[i + kx], w.x);
                        fma2(acc[i][1], d[i + kx], w.y);
                    }
                }
            }
        }
    }

    // ---- the K groups' partials are added in halves (a fixed order); the first group keeps the sum
    auto at = [&](int slab, int i) -> float4* {
        const int R = row * TW + ng * 8 + i;
        return (float4*)(part + (slab * TH * TW + R) * BN + (cg ^ piece<BN, TW>(R)) * 4);
    };
    auto put = [&](int slab) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 lo = halves(acc[i][0]), hi = halves(acc[i][1]);
            *at(slab, i) = make_float4(lo.x, lo.y, hi.x, hi.y);
        }
    };
#pragma unroll 1
    for (int half = KT / 2; half >= 1; half >>= 1) {
        __syncthreads();                                     // every thread is done with the operands / with the slabs before
        if (kt >= half && kt < 2 * half) put(kt - half);
        __syncthreads();
        if (kt < half) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 v = *at(kt, i);
                const float2 lo = halves(acc[i][0]), hi = halves(acc[i][1]);
                acc[i][0] = pair(lo.x + v.x, lo.y + v.y);
                acc[i][1] = pair(hi.x + v.z, hi.y + v.w);
            }
        }
    }
    if (kt == 0) put(0);                                     // (where it has just read itself)
    // ---- row R of the tile's TH x TW belongs to CTA R / rpo of the cluster
    const int rpo = TH * TW / S;
    if (S > 1) {
        if (kt == 0) fence_proxy_async_smem();
        __syncthreads();
        cluster_wait();
        if (tid < S)
            copy_to_peer(map_to_cta(smem_u32(rx + rank * rpo * BN), (uint32_t)tid), smem_u32(part + tid * rpo * BN), (uint32_t)(rpo * BN * 4),
                         map_to_cta(smem_u32(&bars->rx_full), (uint32_t)tid));
        __syncwarp();
    } else {
        rx = part;
        __syncthreads();
    }
    finish_rows<BN, 2>(a, [&](int s, int local, int c) { return rx + (s * rpo + local) * BN + (c ^ piece<BN, TW>(rank * rpo + local)) * 4; }, S, rpo, tid, frame, n0, KIND == KPHASE ? 2 * H : H, KIND == KPHASE ? 2 * W : W,
                        (KIND == KPHASE ? tile * 4 + par : tile) * S + rank,
                        [&](int local, int& oy, int& ox) -> bool {
                            const int R = rank * rpo + local;
                            oy = ty + R / TW;
                            ox = tx + R % TW;
                            const bool valid = oy < H && ox < W;
                            if (KIND == KPHASE) { oy = 2 * oy + (par >> 1); ox = 2 * ox + (par & 1); }
                            return valid;
                        },
                        [&] {
                            if (S > 1) {
                                (void)wait_cluster(smem_u32(&bars->rx_full), 0, abort_flag);
                                __syncwarp();
                                cluster_arrive();            // what is sent to this CTA has landed
                            }
                        });
    if (tid == 0 && bars->abort_flag) {
        land_loads(bars->w_full, n_w, bars->issued);
        if (status && atomicCAS(status, 0u, kStatusConvTimeout) == 0u) {
            status[1] = blockIdx.x;
            status[2] = (uint32_t)BN;
        }
    }
    if (S > 1) {                                             // the sources of this CTA's copies may go
        __syncwarp();
        cluster_wait();
    }
}

// [16 taps][Cin][Cout]: parity * 4 + dy * 2 + dx, each the sum of the 3x3 taps that read the same source pixel (see conv_tc.cu)
template <typename T>
__global__ void pack_weight_f32_phase_kernel(const T* w, float* packed, int Cout, int Cin) {
    const int64_t total = (int64_t)16 * Cout * Cin;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(i % Cout), c = (int)((i / Cout) % Cin), tap = (int)(i / ((int64_t)Cin * Cout));
        const int pa = tap >> 3, pb = (tap >> 2) & 1, dy = (tap >> 1) & 1, dx = tap & 1;
        const int ky0 = dy == 0 ? 0 : 1 + pa, ky1 = dy == 0 ? pa : 2, kx0 = dx == 0 ? 0 : 1 + pb, kx1 = dx == 0 ? pb : 2;
        float v = 0.f;
        for (int ky = ky0; ky <= ky1; ++ky)
            for (int kx = kx0; kx <= kx1; ++kx) {
                const size_t j = ((size_t)o * Cin + c) * 9 + ky * 3 + kx;
                v += sizeof(T) == 2 ? __bfloat162float(((const __nv_bfloat16*)w)[j]) : ((const float*)w)[j];
            }
        packed[i] = v;
    }
}

template <int TH, int BN, int KIND, int TW = 8>
int ops_floats(int n_w) {                                    // operand stages; the partials lie over them
    using C = FCfg<TH, BN, KIND, TW>;
    return std::max((2 * C::IN_FLOATS + 31) / 32 * 32 + n_w * C::W_FLOATS, C::PART_FLOATS);
}
template <int TH, int BN, int KIND, int TW = 8>
int smem_bytes(int n_w, int splits) {
    using C = FCfg<TH, BN, KIND, TW>;
    return (ops_floats<TH, BN, KIND, TW>(n_w) + (splits > 1 ? C::RX_FLOATS : 0)) * 4 + kFTail + 128;
}

template <int TH, int BN, int KIND, int TW = 8>
cudaError_t launch_one(const ConvArgs& a, const ConvF32Plan& p, unsigned int* status, cudaStream_t s) {
    const int H = KIND == KPHASE ? a.Hs : a.H, W = KIND == KPHASE ? a.Ws : a.W;
    const long long ctas = (long long)((W + TW - 1) / TW) * ((H + TH - 1) / TH) * (BN < 32 ? 1 : a.Cout / BN) * (KIND == KPHASE ? 4 : 1) * a.B * p.splits;
    return launch_clusters<conv_f32_kernel<TH, BN, KIND, TW>>({ctas, kThreads, smem_bytes<TH, BN, KIND, TW>(p.n_w, p.splits), kSplitSmemMax, p.splits}, s,
                                                              a, p.splits, p.n_w, ops_floats<TH, BN, KIND, TW>(p.n_w), *(const CUtensorMap*)p.tmap, status);
}

int kind_of(const ConvArgs& a) { return a.upsample == 2 ? KPHASE : (a.ksize == 1 ? K1X1 : K3X3); }

}  // namespace

// The input is read as float4, and outside the frame head so are bias and residual, and the output is written so; the
// weights come by bulk tensor loads.  Layers whose tensors are not aligned for that stay on the direct kernel, and so do
// inputs of more channels than a cluster's slices hold and frames whose pixels or four-channel pieces the kernel's 32-bit
// indices do not reach.  What is supported here has a plan (conv_f32_choose).
bool conv_f32_supported(const ConvArgs& a) {
    if (a.in_dtype != VD_F32 || (a.ksize != 1 && a.ksize != 3) || a.Cin % 4 != 0 || a.x2 || a.upsample == 1) return false;
    if (!aligned16(a.x) || a.Cin > kMaxSplits * kMaxSlice) return false;
    const long long pixels = (long long)a.Hs * a.Ws;
    if (pixels > 0x7fffffffLL || pixels * (a.Cin / 4) > 0xffffffffLL) return false;
    if (a.Cout % 32 == 0 && !(aligned16(a.w) && aligned16(a.bias) && aligned16(a.residual) && aligned16(a.y))) return false;
    if (a.upsample == 2) return a.ksize == 3 && a.Cout % 32 == 0 && !a.out_nchw && !a.out_u8 && a.out_dtype == VD_F32;
    if (a.Cout % 32 == 0) return !a.out_nchw && !a.out_u8 && a.out_dtype == VD_F32;
    // the frame head: its slice of the weights stays in shared memory
    return a.Cout <= 4 && a.ksize == 3 && a.Cin <= 512 && (a.out_nchw || a.out_u8) && !a.residual;
}

// Tile height 8 where 16 would be more than an eighth padding; K divided among a cluster as long as two CTAs per SM are
// not exceeded (a CTA's time is proportional to its share of K, and below that the other SMs idle: 512->512 at 8x8 is 16
// CTAs undivided).
bool conv_f32_choose(const ConvArgs& a, ConvF32Plan* p, int max_splits) {
    p->valid = 0;
    if (!conv_f32_supported(a)) return false;
    const int kind = kind_of(a);
    const bool head = a.Cout % 32 != 0;
    const int H = kind == KPHASE ? a.Hs : a.H, W = kind == KPHASE ? a.Ws : a.W;
    const int rows8 = (H + 7) / 8 * 8, rows16 = (H + 15) / 16 * 16;
    p->th = !head && rows16 * 7 > rows8 * 8 ? 8 : 16;
    p->bn = head ? 4 : 32;
    // the frame head of a large image: tiles 32 pixels wide (see FCfg), unless they are more than half padding
    const long long wide = (long long)((W + 31) / 32) * ((H + 15) / 16);
    p->tw = head && wide * std::max(a.B, 1) >= 148 && (W + 31) / 32 * 2 <= (W + 7) / 8 ? 32 : 8;
    const int tiles = ((W + p->tw - 1) / p->tw) * ((H + p->th - 1) / p->th), chunks = (a.Cin + kChunk - 1) / kChunk;
    const long long ctas = (long long)tiles * (head ? 1 : a.Cout / 32) * (kind == KPHASE ? 4 : 1) * std::max(a.B, 1);
    int s = 1;
    while (s < max_splits && 2 * s <= chunks && ctas * 2 * s <= 296) s *= 2;
    while ((chunks + s - 1) / s * kChunk > (head ? 128 : kMaxSlice)) s *= 2;
    if (s > max_splits) return false;
    p->splits = s;
    const int units = (chunks + s - 1) / s;
    auto fit = [&](int base, int stage) { return std::min(std::min(units, kMaxW), (kSplitSmemMax - base) / stage); };
    if (head) p->n_w = units;
    else if (p->th == 16) {
        p->n_w = kind == K3X3 ? fit(smem_bytes<16, 32, K3X3>(0, s), FCfg<16, 32, K3X3>::W_FLOATS * 4)
                 : kind == K1X1 ? fit(smem_bytes<16, 32, K1X1>(0, s), FCfg<16, 32, K1X1>::W_FLOATS * 4)
                                : fit(smem_bytes<16, 32, KPHASE>(0, s), FCfg<16, 32, KPHASE>::W_FLOATS * 4);
    } else {
        p->n_w = kind == K3X3 ? fit(smem_bytes<8, 32, K3X3>(0, s), FCfg<8, 32, K3X3>::W_FLOATS * 4)
                 : kind == K1X1 ? fit(smem_bytes<8, 32, K1X1>(0, s), FCfg<8, 32, K1X1>::W_FLOATS * 4)
                                : fit(smem_bytes<8, 32, KPHASE>(0, s), FCfg<8, 32, KPHASE>::W_FLOATS * 4);
    }
    return p->n_w >= 1;
}

int conv_f32_slots(const ConvArgs& a, const ConvF32Plan& p, int groups) {
    const int H = a.upsample == 2 ? a.Hs : a.H, W = a.upsample == 2 ? a.Ws : a.W;
    return ((W + p.tw - 1) / p.tw) * ((H + p.th - 1) / p.th) * (a.upsample == 2 ? 4 : 1) * p.splits * rec_parts(p.bn, a.Cout / groups);
}

cudaError_t conv_f32_prepare(const ConvArgs& a, ConvF32Plan* p) {
    if (p->bn == 32) {
        EncodeTiledFn enc = encode_fn();
        if (!enc) return cudaErrorNotSupported;
        const int taps = a.upsample == 2 ? 16 : a.ksize * a.ksize;
        const cuuint64_t d[3] = {(cuuint64_t)a.Cout, (cuuint64_t)a.Cin, (cuuint64_t)taps};
        const cuuint64_t st[2] = {(cuuint64_t)a.Cout * 4, (cuuint64_t)a.Cout * a.Cin * 4};
        const cuuint32_t box[3] = {32, kChunk, (cuuint32_t)(a.upsample == 2 ? 4 : taps)};
        const cuuint32_t one[3] = {1, 1, 1};
        if (enc((CUtensorMap*)p->tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(a.w), d, st, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    p->valid = 1;
    return cudaSuccess;
}

// f(Build<...>) for the build that the plan takes
namespace {
template <int TH, int BN, int KIND, int TW = 8> struct Build {
    static cudaError_t launch(const ConvArgs& a, const ConvF32Plan& p, unsigned int* status, cudaStream_t s) { return launch_one<TH, BN, KIND, TW>(a, p, status, s); }
    static bool fits(const ConvF32Plan& p) { return clusters_fit<conv_f32_kernel<TH, BN, KIND, TW>>(kThreads, kSplitSmemMax, p.splits); }
};
template <class F> auto with_build(const ConvArgs& a, const ConvF32Plan& p, F f) {
    const int kind = kind_of(a);
    if (p.bn == 4) return p.tw == 32 ? f(Build<16, 4, K3X3, 32>()) : f(Build<16, 4, K3X3>());
    if (p.th == 8) {
        if (kind == K3X3) return f(Build<8, 32, K3X3>());
        return kind == K1X1 ? f(Build<8, 32, K1X1>()) : f(Build<8, 32, KPHASE>());
    }
    if (kind == K3X3) return f(Build<16, 32, K3X3>());
    return kind == K1X1 ? f(Build<16, 32, K1X1>()) : f(Build<16, 32, KPHASE>());
}
}  // namespace

bool conv_f32_fits(const ConvArgs& a, const ConvF32Plan& p) {
    return with_build(a, p, [&](auto build) { return build.fits(p); });
}

cudaError_t launch_conv_f32(const ConvArgs& a, const ConvF32Plan& p, unsigned int* status, cudaStream_t s) {
    if (!p.valid) return cudaErrorInvalidValue;
    if (a.in_rec && !rec_groups_ok(a.Cin, a.in_G)) return cudaErrorInvalidValue;
    if (a.out_rec && !rec_groups_ok(a.Cout, a.out_G)) return cudaErrorInvalidValue;
    return with_build(a, p, [&](auto build) { return build.launch(a, p, status, s); });
}

cudaError_t launch_pack_weight_f32_phase(const void* w, int w_dtype, float* packed, int Cout, int Cin, cudaStream_t s) {
    const int grid = (int)std::min<int64_t>(((int64_t)16 * Cout * Cin + 255) / 256, 148 * 16);
    if (w_dtype == VD_BF16) pack_weight_f32_phase_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>((const __nv_bfloat16*)w, packed, Cout, Cin);
    else pack_weight_f32_phase_kernel<float><<<grid, 256, 0, s>>>((const float*)w, packed, Cout, Cin);
    return cudaGetLastError();
}

// One block per (group, frame) merges a layer's records into scale and shift: where there are too many for every CTA of
// the consuming layer to merge for itself, or the consumer cannot.
namespace {
constexpr int kMergeThreads = 512;
__global__ void __launch_bounds__(kMergeThreads) gn_merge_kernel(GnArgs a) {
    __shared__ float2 s_part[kMergeThreads / 32];
    griddep_launch();
    const int g = blockIdx.x, n = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cpg = a.C / a.G, c = g * cpg + threadIdx.x;
    const bool mine = threadIdx.x < cpg;
    const float gamma = mine ? __ldg(a.gamma + c) : 0.f, beta = mine ? __ldg(a.beta + c) : 0.f, off = mine && a.offset ? __ldg(a.offset + c) : 0.f;
    const float4* rec = a.rec + ((size_t)n * a.G + g) * a.slots;
    griddep_wait();
    const float ref = __ldcg(&rec->y);
    float s = 0.f, q = 0.f;
    constexpr int U = 8;                                     // records of a thread on their way at a time
    for (int i0 = threadIdx.x; i0 < a.slots; i0 += U * kMergeThreads) {
        float4 r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) r[u] = i0 + u * kMergeThreads < a.slots ? __ldcg(rec + i0 + u * kMergeThreads) : make_float4(0.f, ref, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float d = r[u].y - ref, nd = r[u].x * d;
            s += nd;
            q += fmaf(nd, d, r[u].z);
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, d);
        q += __shfl_xor_sync(0xffffffffu, q, d);
    }
    if (lane == 0) s_part[warp] = make_float2(s, q);
    __syncthreads();
    if (!mine) return;
    float2 t = s_part[0];
#pragma unroll
    for (int w = 1; w < kMergeThreads / 32; ++w) { t.x += s_part[w].x; t.y += s_part[w].y; }
    const float inv_n = 1.f / ((float)a.P * (float)cpg), dm = t.x * inv_n;
    const float sc = gamma * (1.f / sqrtf(fmaxf(fmaf(-dm, dm, t.y * inv_n), 0.f) + a.eps));
    a.scale[(size_t)n * a.C + c] = sc;
    a.shift[(size_t)n * a.C + c] = beta - (ref + dm - off) * sc;
}
}  // namespace
cudaError_t launch_gn_merge(const GnArgs& a, cudaStream_t s) {
    if (a.C / a.G > kMergeThreads) return cudaErrorInvalidValue;
    return launch_pdl(gn_merge_kernel, dim3(a.G, a.B), dim3(kMergeThreads), 0, s, a);
}

}  // namespace vd
