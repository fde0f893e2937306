// Shared by the convolution kernels whose CTAs divide K among a thread-block cluster (conv_f32.cu, conv_split.cu):
// the exchange of partial sums through distributed shared memory, and GroupNorm statistics as records.
//
//   * A CTA adds up and writes 1/S of its cluster's output rows (row = pixel of the tile).  Every CTA lays its partials
//     out in its own shared memory, and bulk copies carry an owner's rows there and count the bytes on the owner's barrier:
//     one wait, no cluster-wide barrier on the way.  (16-byte st.async stores straight from registers
//     took 2.3-3.7 us of a 12 us layer: 2048 packets per CTA.)  The owner adds the partials in a fixed order (bitwise
//     reproducible).
//   * While it writes its rows a CTA takes their statistics, and leaves one record (count, mean, sum of squared
//     deviations) per group and warp share.  The CTAs of the layer that normalises merge the records of their own input
//     channels (Chan's formula, a fixed order), or a small launch does where there are many.  The normalisation then
//     costs neither a read of the tensor nor, mostly, a launch.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include <mutex>

#include "tc_common.cuh"
#include "tc_pair.cuh"
#include "vd_internal.h"

namespace vd {
namespace cc {

constexpr int kFinishThreads = 256;                          // eight warps add up and write the rows

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
// Bounded like mbar_wait, for data that other CTAs of the cluster send.  It does not return early when a wait of this CTA has
// already given up: the others send theirs all the same, and it must not land in shared memory that is gone.
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag) {
    if (try_wait_cluster(bar, parity)) return true;
    const long long t0 = clock64();
    while (!try_wait_cluster(bar, parity))
        if (clock64() - t0 > tc::WAIT_LIMIT_CYCLES) { *abort_flag = 1; return false; }
    return true;
}

// Where a wait gave up, loads into shared memory may still be on their way when everybody else is done: load k of `issued`
// (into stage k % stages, counted on that stage's barrier) has landed when this returns, or the limit has passed.  Out of line:
// as part of the kernels its code cost 0.4 % of the smallest fp32 call (127.0 -> 127.5 us, 126.3 so).
static __device__ __noinline__ void land_loads(const uint64_t* full, int stages, int issued) {
    for (int k = max(issued - stages, 0); k < issued; ++k) {
        const long long t0 = clock64();
        while (!tc::mbar_try_wait(tc::smem_u32(full + k % stages), (k / stages) & 1) && clock64() - t0 < tc::WAIT_LIMIT_CYCLES) {}
    }
}

// The launch's parameters come through the constant cache, a line at a time: one warp reads a word of every line while the
// kernel before is still running, so that nobody waits for the first use of one later.  (The sum goes to an unused word of
// shared memory, or nothing would be read.)
__device__ __forceinline__ void touch_params(const ConvArgs& a, volatile uint32_t* unused) {
    *unused = (uint32_t)(size_t)a.bias + (uint32_t)(size_t)a.y + (uint32_t)a.out_dtype + (uint32_t)(size_t)a.bias2 + (uint32_t)(size_t)a.stat_gamma +
              __float_as_uint(a.stat_eps) + (uint32_t)a.in_slots + __float_as_uint(a.in_inv_n) + (uint32_t)(size_t)a.out_rec + (uint32_t)a.out_shift + (uint32_t)a.silu + a.div_tx;
}

// half * scale and half * shift of the input channels [c0, c0 + nch) of `frame`, from the producing layer's records, by
// NW warps (w = 0..NW - 1); c0 and nch are multiples of the group size.  A group has 8 lanes of a warp (32 where there are more
// than 16 records); a lane's first NR records are loaded by `load`, so that they are on their way before other loads, and
// `finish` merges.  Deviations are from the first record's mean, so one round of loads and one of shuffles suffice.
// Everything that does not need the kernel before is done ahead by `prepare`, gamma and beta into s_scale and s_shift
// included (a lane reads back what it has put there itself); what stays in registers across the loads is kept small, since
// a loaded value that is spilled has to be waited for.
template <int NW, int NR> struct InputStatsOf {
    const float4* rec;
    float4 r[NR];
    int g;                                                   // this lane's group of the slice
    static __device__ __forceinline__ int lanes_log2(const ConvArgs& a) { return a.in_slots <= 16 ? 3 : 5; }
    __device__ __forceinline__ void prepare(const ConvArgs& a, int frame, int c0, int nch, int w, int lane, float* s_scale, float* s_shift) {
        const int ll = lanes_log2(a), L = 1 << ll, l = lane & (L - 1), ng = nch >> a.in_shift;
        g = (w << (5 - ll)) + (lane >> ll);
        rec = a.in_rec + ((size_t)frame * a.in_G + (c0 >> a.in_shift) + min(g, ng - 1)) * a.in_slots;
#pragma unroll 1
        for (int gg = g; gg < ng; gg += NW << (5 - ll))
            for (int i = l; i < 1 << a.in_shift; i += L) {
                const int c = (gg << a.in_shift) + i;
                s_scale[c] = __ldg(a.in_gamma + c0 + c);
                s_shift[c] = __ldg(a.in_beta + c0 + c);
            }
    }
    __device__ __forceinline__ void load(const ConvArgs& a, int lane) {
        const int ll = lanes_log2(a), L = 1 << ll, l = lane & (L - 1);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            r[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (l + i * L < a.in_slots) r[i] = __ldcg(rec + l + i * L);
        }
    }
    __device__ __forceinline__ void finish(const ConvArgs& a, int nch, int lane, float half, float* s_scale, float* s_shift) {
        const int ll = lanes_log2(a), L = 1 << ll, l = lane & (L - 1), ng = nch >> a.in_shift;
#pragma unroll 1
        for (;;) {
            const float ref = __shfl_sync(0xffffffffu, r[0].y, lane & ~(L - 1));
            float s = 0.f, q = 0.f;
            auto add = [&](const float4& v) {
                const float d = v.y - ref, nd = v.x * d;
                s += nd;
                q += fmaf(nd, d, v.z);
            };
#pragma unroll
            for (int i = 0; i < NR; ++i) add(r[i]);
#pragma unroll 1
            for (int i = l + NR * L; i < a.in_slots; i += L) add(__ldcg(rec + i));
            if (ll == 5) {
                s += __shfl_xor_sync(0xffffffffu, s, 16); q += __shfl_xor_sync(0xffffffffu, q, 16);
                s += __shfl_xor_sync(0xffffffffu, s, 8); q += __shfl_xor_sync(0xffffffffu, q, 8);
            }
#pragma unroll
            for (int d = 4; d > 0; d >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, d);
                q += __shfl_xor_sync(0xffffffffu, q, d);
            }
            const float dm = s * a.in_inv_n, mean = ref + dm;
            const float rstd = 1.f / sqrtf(fmaxf(fmaf(-dm, dm, q * a.in_inv_n), 0.f) + a.in_eps);
            if (g < ng)
                for (int i = l; i < 1 << a.in_shift; i += L) {
                    const int c = (g << a.in_shift) + i;
                    const float sc = s_scale[c] * rstd;
                    s_scale[c] = sc * half;
                    s_shift[c] = (s_shift[c] - mean * sc) * half;
                }
            const int step = NW << (5 - ll);
            if (g - (lane >> ll) + step >= ng) break;        // (the same for the whole warp)
            rec += (size_t)(min(g + step, ng - 1) - min(g, ng - 1)) * a.in_slots;
            g += step;
            load(a, lane);
        }
    }
};
using InputStats = InputStatsOf<8, 2>;

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
// records.  source(s, row, c): where channels [4c, 4c + 4) of row `row` of partial s lie.  ptid: 0..255.
// locate(local row, oy, ox) gives the row's output pixel and whether it exists; ready() returns when the partials have
// arrived.  The first PRE rows' addresses and residual and the record's address are made before that (the empty asm keeps
// them there).
// A thread takes four channels (cg) of every RSTEP-th row, so a warp's share of a group comes from shuffles alone.  BN < 32:
// the frame head (planes or packed pixels of a.Cout channels).
template <int BN, int PRE, class Source, class Locate, class Ready>
__device__ __forceinline__ void finish_rows(const ConvArgs& a, Source source, int nparts, int rpo, int ptid, int frame, int n0, int OH, int OW,
                                            int slot0, Locate locate, Ready ready) {
    constexpr bool HEAD = BN < 32;
    constexpr int CPW = HEAD ? 1 : Split8<HEAD ? 64 : BN>::CPW, WC = HEAD ? 1 : Split8<HEAD ? 64 : BN>::WC, RL = 32 / CPW;
    constexpr int RSTEP = HEAD ? kFinishThreads / (BN / 4) : RL * (8 / WC), CPW_LOG2 = CPW == 8 ? 3 : CPW == 4 ? 2 : CPW - 1;
    static_assert(CPW == 1 || CPW == 2 || CPW == 4 || CPW == 8, "columns of a warp");
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
    float4 res[PRE];
    size_t off[PRE];                                         // element of y (head: pixel of the frame)
    bool valid[PRE];
    auto place = [&](int first) {
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            res[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            int oy = 0, ox = 0;
            valid[i] = first + i * RSTEP < rpo && locate(first + i * RSTEP, oy, ox);
            off[i] = HEAD ? (size_t)oy * OW + ox : (((size_t)frame * OH + oy) * OW + ox) * a.Cout + co;
            asm volatile("" : "+l"(off[i]));
            if (!HEAD && a.residual && valid[i]) res[i] = __ldcg((const float4*)(a.residual + off[i]));
        }
    };
    place(rg);
    // statistics: deviations from a value of the group (the first one inside the image that this warp holds)
    const int side_log2 = max(a.out_shift - 2 - CPW_LOG2, 0), part = ((w / WC) << side_log2) + ((w % WC) & ((1 << side_log2) - 1));
    const int peer_lanes = RL << min(max(a.out_shift - 2, 0), CPW_LOG2);
    uint32_t peers = (0xffffffffu >> (32 - peer_lanes)) << (lane & -peer_lanes & 31);
    float4* rec = a.out_rec + ((size_t)frame * a.out_G + (co >> a.out_shift)) * a.out_slots + ((slot0 * (8 / WC)) << side_log2) + part;
    asm volatile("" : "+l"(rec), "+r"(peers));
    ready();
    float sum = 0.f, sq = 0.f, pivot = 0.f;
    int cnt = 0;
#pragma unroll 1
    for (int l0 = rg - lane % RL; l0 < rpo; l0 += PRE * RSTEP) {
        const int first = l0 + lane % RL;
        if (first != rg) place(first);
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            const int local = first + i * RSTEP;
            float4 v = bias;
            if (valid[i]) {
#pragma unroll 4
                for (int s = 0; s < nparts; ++s) {
                    const float4 p = *(const float4*)source(s, local, cg);
                    v.x += p.x; v.y += p.y; v.z += p.z; v.w += p.w;
                }
                if (HEAD) {
                    const float f[4] = {v.x, v.y, v.z, v.w};
                    const size_t plane = (size_t)OH * OW;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (co + e >= a.Cout) break;
                        const float x = f[e] + (a.bias ? __ldg(a.bias + co + e) : 0.f);
                        const size_t o = ((size_t)frame * a.Cout + co + e) * plane + off[i];
                        if (a.out_u8) ((unsigned char*)a.y)[(frame * plane + off[i]) * a.Cout + co + e] = pack_u8(x);
                        else if (a.out_dtype == VD_BF16) ((__nv_bfloat16*)a.y)[o] = __float2bfloat16_rn(x);
                        else ((float*)a.y)[o] = x;
                    }
                } else if (a.out_dtype == VD_BF16) {
                    const uint32_t lo = tc::pack_bf16(v.x, v.y), hi = tc::pack_bf16(v.z, v.w);
                    *(uint2*)((__nv_bfloat16*)a.y + off[i]) = make_uint2(lo, hi);
                    v = make_float4(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u), __uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
                } else {
                    v.x += res[i].x; v.y += res[i].y; v.z += res[i].z; v.w += res[i].w;
                    *(float4*)((float*)a.y + off[i]) = v;
                }
            }
            if (!HEAD && a.out_rec) {
                const uint32_t m = __ballot_sync(0xffffffffu, valid[i]) & peers;
                if (l0 + i * RSTEP < RSTEP)                  // the warp's first rows
                    pivot = __shfl_sync(0xffffffffu, v.x, m ? __ffs(m) - 1 : lane);
                cnt += __popc(m);
                if (valid[i]) {
                    const float d0 = v.x - pivot, d1 = v.y - pivot, d2 = v.z - pivot, d3 = v.w - pivot;
                    sum += (d0 + d1) + (d2 + d3);
                    sq += fmaf(d0, d0, d1 * d1) + fmaf(d2, d2, d3 * d3);
                }
            }
        }
    }
    if (!HEAD && a.out_rec) {
        const float n = (float)(cnt * 4), inv = cnt ? 1.f / n : 0.f;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1)
            if (d < RL || d < peer_lanes) {
                sum += __shfl_xor_sync(0xffffffffu, sum, d);
                sq += __shfl_xor_sync(0xffffffffu, sq, d);
            }
        if ((lane & (peer_lanes - 1)) == 0) {
            const float dm = sum * inv;
            *rec = make_float4(n, pivot + dm, fmaxf(fmaf(-dm, sum, sq), 0.f), 0.f);
        }
    }
}

// ---- launches of kernels that run as clusters
// `smem_max`: the kernel's shared-memory limit, set once per device.
constexpr int kMaxDevices = 64;
template <auto KERNEL> cudaError_t set_smem_limit(int smem_max) {
    static std::mutex mu;
    static bool done[kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!done[dev]) {
        e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        if (e != cudaSuccess) return e;
        done[dev] = true;
    }
    return cudaSuccess;
}
// Can the current device hold a cluster of `cluster` such CTAs at all?  (A part of a GPU may have too few SMs side by side.)
// Asked once per device and size, for the largest shared memory that the kernel is launched with.
template <auto KERNEL> bool clusters_fit(int threads, int smem_max, int cluster) {
    static std::mutex mu;
    static signed char known[kMaxDevices][4] = {};           // by log2 of the size: 0 not asked, 1 yes, -1 no
    int dev = 0, l = 0;
    while (1 << l < cluster) ++l;
    if (l == 0) return true;
    if (l > 3 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices || set_smem_limit<KERNEL>(smem_max) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!known[dev][l]) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)cluster);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = (size_t)smem_max;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, (const void*)KERNEL, &cfg);
        if (e != cudaSuccess) cudaGetLastError();
        known[dev][l] = e == cudaSuccess && n > 0 ? 1 : -1;
    }
    return known[dev][l] > 0;
}
struct ClusterShape { long long ctas; int threads, smem, smem_max, cluster; };
template <auto KERNEL, class... Args> cudaError_t launch_clusters(const ClusterShape& c, cudaStream_t s, Args&&... args) {
    cudaError_t e = set_smem_limit<KERNEL>(c.smem_max);
    if (e != cudaSuccess) return e;
    if (c.ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)c.ctas);
    cfg.blockDim = dim3((unsigned)c.threads);
    cfg.dynamicSmemBytes = (size_t)c.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)c.cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, KERNEL, std::forward<Args>(args)...);
}

}  // namespace cc
}  // namespace vd
