// Shared by the convolution kernels whose CTAs divide K among a thread-block cluster (conv_f32.cu, conv_split.cu):
// the exchange of partial sums through distributed shared memory, and GroupNorm statistics as records.
//
//   * A CTA adds up and writes 1/S of its cluster's output rows (row = pixel of the tile).  Every CTA lays its partials
//     out in its own shared memory, and one bulk copy per owner carries an owner's rows there and counts the bytes on the
//     owner's barrier: one wait, no cluster-wide barrier on the way.  (16-byte st.async stores straight from registers
//     took 2.3-3.7 us of a 12 us layer: 2048 packets per CTA.)  The owner adds the partials in a fixed order (bitwise
//     reproducible).
//   * While it writes its rows a CTA takes their statistics, and leaves one record (count, mean, sum of squared
//     deviations) per group and warp share.  The CTAs of the layer that normalises merge the records of their own input
//     channels (Chan's formula, a fixed order), or a small launch does where there are many.  The normalisation then
//     costs neither a read of the tensor nor, mostly, a launch.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "tc_common.cuh"
#include "vd_internal.h"

namespace vd {
namespace cc {

constexpr int kFinishThreads = 256;                          // eight warps add up and write the rows

__device__ __forceinline__ uint32_t ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t smem_addr, uint32_t cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(cta));
    return r;
}
// `bytes` (a multiple of 16) from this CTA's shared memory into another CTA's (cluster addresses); their arrival is
// counted on that CTA's barrier `bar`
__device__ __forceinline__ void copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0u;
}
// bounded like mbar_wait, for data that other CTAs of the cluster have stored
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag) {
    if (try_wait_cluster(bar, parity)) return true;
    const long long t0 = clock64();
    while (!try_wait_cluster(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > tc::WAIT_LIMIT_CYCLES) { *abort_flag = 1; return false; }
    }
    return true;
}

// Statistics of one group from its records (count, mean, sum of squared deviations), for the whole warp the same number L
// (8 or 32) of lanes to a group.  Deviations are from the first record's mean, so one round of loads and one of shuffles
// suffice; a lane's first two records are loaded by `load`, so that they are on their way before other loads.
struct GroupRecords {
    float4 r0, r1;
    float ref;
    __device__ __forceinline__ void load(const float4* rec, int slots, int l, int L) {
        ref = __ldcg(&rec->y);
        r0 = r1 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (l < slots) r0 = __ldcg(rec + l);
        if (l + L < slots) r1 = __ldcg(rec + l + L);
    }
    __device__ __forceinline__ void merge(const float4* rec, int slots, int l, int L, float inv_n, float eps, float& mean, float& rstd) const {
        const float d0 = r0.y - ref, d1 = r1.y - ref, n0 = r0.x * d0, n1 = r1.x * d1;
        float s = n0 + n1, q = fmaf(n0, d0, r0.z) + fmaf(n1, d1, r1.z);
        for (int i = l + 2 * L; i < slots; i += L) {
            const float4 r = __ldcg(rec + i);
            const float d = r.y - ref, nd = r.x * d;
            s += nd;
            q += fmaf(nd, d, r.z);
        }
        for (int d = L >> 1; d > 0; d >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, d);
            q += __shfl_xor_sync(0xffffffffu, q, d);
        }
        const float dm = s * inv_n;
        mean = ref + dm;
        rstd = 1.f / sqrtf(fmaxf(fmaf(-dm, dm, q * inv_n), 0.f) + eps);
    }
};

// half * scale and half * shift of the input channels [c0, c0 + nch) of `frame`, from the producing layer's records, by
// NW warps (w = 0..NW - 1); c0 and nch are multiples of the group size.  Everything but the records is ready before
// the kernel before has finished: set up with `prepare`, then `load`, then (other loads issued) `finish`.
template <int NW> struct InputStatsOf {
    const float4* rec;
    int cpg, L, l, g, ng;
    float inv_n, gamma[2], beta[2];
    GroupRecords gr;
    __device__ __forceinline__ void prepare(const ConvArgs& a, int frame, int c0, int nch, int w, int lane) {
        cpg = a.Cin / a.in_G;
        L = a.in_slots <= 16 ? 8 : 32;
        l = lane & (L - 1);
        ng = nch / cpg;
        g = w * (32 / L) + lane / L;
        inv_n = 1.f / ((float)a.in_pixels * (float)cpg);
        rec = a.in_rec + ((size_t)frame * a.in_G + c0 / cpg + min(g, ng - 1)) * a.in_slots;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int c = c0 + min(g, ng - 1) * cpg + l + i * L;
            const bool on = l + i * L < cpg;
            gamma[i] = on ? __ldg(a.in_gamma + c) : 0.f;
            beta[i] = on ? __ldg(a.in_beta + c) : 0.f;
        }
    }
    __device__ __forceinline__ void load(const ConvArgs& a) { gr.load(rec, a.in_slots, l, L); }
    __device__ __forceinline__ void finish(const ConvArgs& a, int c0, float half, float* s_scale, float* s_shift) {
        const int step = NW * (32 / L);
        for (;;) {
            float mean, rstd;
            gr.merge(rec, a.in_slots, l, L, inv_n, a.in_eps, mean, rstd);
            if (g < ng) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (l + i * L < cpg) {
                        const float sc = gamma[i] * rstd;
                        s_scale[g * cpg + l + i * L] = sc * half;
                        s_shift[g * cpg + l + i * L] = (beta[i] - mean * sc) * half;
                    }
            }
            if (g - (int)(threadIdx.x & 31) / L + step >= ng) break;     // (the same for the whole warp)
            g += step;
            rec += (size_t)step * a.in_slots;
            const int gg = min(g, ng - 1);
            rec -= (size_t)(g - gg) * a.in_slots;
            gr.load(rec, a.in_slots, l, L);
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (l + i * L < cpg) {
                    gamma[i] = __ldg(a.in_gamma + c0 + gg * cpg + l + i * L);
                    beta[i] = __ldg(a.in_beta + c0 + gg * cpg + l + i * L);
                }
        }
    }
};

using InputStats = InputStatsOf<8>;

// The eight warps that write a CTA's rows: a warp has CPW four-channel columns of the BN channels (two at least: whole
// 32-byte sectors), WC warps lie side by side and WR below one another.
template <int BN> struct Split8 {
    static constexpr int CPW = BN / 32 > 2 ? BN / 32 : 2, WC = BN / (4 * CPW), WR = 8 / WC;
};
// records that a CTA leaves per group of `cpg` channels (4, 8 or 16)
inline int rec_parts(int bn, int cpg) {
    const int cpw = bn / 32 > 2 ? bn / 32 : 2;
    return (cpg > 4 * cpw ? cpg / (4 * cpw) : 1) * (8 / (bn / (4 * cpw)));
}

// Adds up the `nparts` partials of this CTA's `rpo` rows, adds bias and residual, writes the output and the statistics
// records.  rx: [nparts][rpo][RXS] floats, 16-byte piece c of a row at c ^ swizzle(row).  ptid: 0..255.  locate(local row, oy, ox) gives the row's output pixel and
// whether it exists; ready() returns when the partials have arrived (the residual is on its way by then).
// A thread takes four channels (cg) of every RSTEP-th row, so a warp's share of a group comes from shuffles alone.  BN < 32: the frame head (planes or packed pixels of a.Cout channels).
template <int BN, int RXS, class Locate, class Swizzle, class Ready>
__device__ __forceinline__ void finish_rows(const ConvArgs& a, float* rx, int nparts, int rpo, int ptid, int frame, int n0, int OH, int OW,
                                            int slot0, Locate locate, Swizzle swizzle, Ready ready) {
    constexpr bool HEAD = BN < 32;
    constexpr int CPW = HEAD ? 1 : Split8<HEAD ? 64 : BN>::CPW, WC = HEAD ? 1 : Split8<HEAD ? 64 : BN>::WC, RL = 32 / CPW;
    constexpr int RSTEP = HEAD ? kFinishThreads / (BN / 4) : RL * (8 / WC);
    const int w = ptid >> 5, lane = ptid & 31;
    const int cg = HEAD ? ptid % (BN / 4) : (w % WC) * CPW + lane / RL, rg = HEAD ? ptid / (BN / 4) : (w / WC) * RL + lane % RL;
    const int co = n0 + cg * 4;
    float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!HEAD) {
        if (a.bias) bias = __ldg((const float4*)(a.bias + co));
        if (a.bias2) {
            const float4 t = __ldg((const float4*)(a.bias2 + co));
            bias.x += t.x; bias.y += t.y; bias.z += t.z; bias.w += t.w;
        }
    }
    constexpr int PRE = 2;                                   // residual rows on their way at a time
    float4 res[PRE];
    auto load_residual = [&](int l0) {
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            res[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            int oy, ox;
            if (!HEAD && a.residual && l0 + i * RSTEP < rpo && locate(l0 + i * RSTEP, oy, ox))
                res[i] = __ldcg((const float4*)(a.residual + (((size_t)frame * OH + oy) * OW + ox) * a.Cout + co));
        }
    };
    load_residual(rg);
    ready();
    // statistics: deviations from a value of the group (the first one inside the image that this warp holds)
    const int cpg = !HEAD && a.out_rec ? a.Cout / a.out_G : 4, lpg = min(cpg >> 2, CPW);        // four-channel columns of a group in this warp
    const uint32_t peers = (lpg * RL >= 32 ? 0xffffffffu : ((1u << (lpg * RL & 31)) - 1u)) << (lane / (lpg * RL) * (lpg * RL));
    float sum = 0.f, sq = 0.f, cnt = 0.f, pivot = 0.f;
#pragma unroll 1
    for (int l0 = rg - lane % RL; l0 < rpo; l0 += PRE * RSTEP) {
        const int first = l0 + lane % RL;
        if (first != rg) load_residual(first);
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            const int local = first + i * RSTEP;
            int oy = 0, ox = 0;
            const bool on = local < rpo, valid = on && locate(local, oy, ox);
            const size_t pixel = ((size_t)frame * OH + oy) * OW + ox;
            float4 v = bias;
            const float* q = rx + local * RXS + (cg ^ swizzle(local)) * 4;
#pragma unroll 4
            for (int s = 0; s < nparts; ++s) {
                if (!on) break;
                const float4 p = *(const float4*)(q + (size_t)s * rpo * RXS);
                v.x += p.x; v.y += p.y; v.z += p.z; v.w += p.w;
            }
            if (valid) {
                if (HEAD) {
                    const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (co + e >= a.Cout) break;
                        const float x = f[e] + (a.bias ? __ldg(a.bias + co + e) : 0.f);
                        const size_t o = (((size_t)frame * a.Cout + co + e) * OH + oy) * OW + ox;
                        if (a.out_u8) ((unsigned char*)a.y)[pixel * a.Cout + co + e] = pack_u8(x);
                        else if (a.out_dtype == VD_BF16) ((__nv_bfloat16*)a.y)[o] = __float2bfloat16_rn(x);
                        else ((float*)a.y)[o] = x;
                    }
                } else if (a.out_dtype == VD_BF16) {
                    const uint32_t lo = tc::pack_bf16(v.x, v.y), hi = tc::pack_bf16(v.z, v.w);
                    *(uint2*)((__nv_bfloat16*)a.y + pixel * a.Cout + co) = make_uint2(lo, hi);
                    v = make_float4(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u), __uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
                } else {
                    v.x += res[i].x; v.y += res[i].y; v.z += res[i].z; v.w += res[i].w;
                    *(float4*)((float*)a.y + pixel * a.Cout + co) = v;
                }
            }
            if (!HEAD && a.out_rec) {
                if (l0 + i * RSTEP < RSTEP) {                // the warp's first rows
                    const uint32_t m = __ballot_sync(0xffffffffu, valid) & peers;
                    pivot = __shfl_sync(0xffffffffu, v.x, m ? __ffs(m) - 1 : lane);
                }
                if (valid) {
                    const float d0 = v.x - pivot, d1 = v.y - pivot, d2 = v.z - pivot, d3 = v.w - pivot;
                    sum += (d0 + d1) + (d2 + d3);
                    sq += fmaf(d0, d0, d1 * d1) + fmaf(d2, d2, d3 * d3);
                    cnt += 4.f;
                }
            }
        }
    }
    if (!HEAD && a.out_rec) {
        for (int d = 1; d < lpg * RL; d <<= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, d);
            sq += __shfl_xor_sync(0xffffffffu, sq, d);
            cnt += __shfl_xor_sync(0xffffffffu, cnt, d);
        }
        if ((lane & (lpg * RL - 1)) == 0) {
            const int side = max(cpg / (4 * CPW), 1), part = (w / WC) * side + (w % WC) % side;
            const float dm = cnt > 0.f ? sum / cnt : 0.f;
            a.out_rec[((size_t)frame * a.out_G + co / cpg) * a.out_slots + slot0 * (side * (8 / WC)) + part] =
                make_float4(cnt, pivot + dm, fmaxf(fmaf(-dm, sum, sq), 0.f), 0.f);
        }
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        return cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess
                   ? (EncodeTiledFn)p : (EncodeTiledFn) nullptr;
    }();
    return fn;
}

}  // namespace cc
}  // namespace vd
