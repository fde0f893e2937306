// Plain FFMA kernels: latent ingest, GroupNorm statistics, a tiled direct convolution with the
// fused prologue/epilogue, a streaming-softmax attention, and weight repacking.  These run the
// fp32 configuration end to end and serve as the on-GPU cross-check path of the bf16 one.
#include <math.h>

#include <mutex>
#include <string>

#include "conv_cluster.cuh"
#include "vd_internal.h"

namespace vd {

namespace {

using namespace tc;

template <typename T> __device__ __forceinline__ float ld_f(const T* p, size_t i);
template <> __device__ __forceinline__ float ld_f<float>(const float* p, size_t i) { return p[i]; }
template <> __device__ __forceinline__ float ld_f<__nv_bfloat16>(const __nv_bfloat16* p, size_t i) {
    return __bfloat162float(p[i]);
}
template <typename T> __device__ __forceinline__ void st_f(T* p, size_t i, float v);
template <> __device__ __forceinline__ void st_f<float>(float* p, size_t i, float v) { p[i] = v; }
template <> __device__ __forceinline__ void st_f<__nv_bfloat16>(__nv_bfloat16* p, size_t i, float v) {
    p[i] = __float2bfloat16_rn(v);
}
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
__device__ __forceinline__ float silu_f(float v) { return v / (1.0f + expf(-v)); }

// ------------------------------------------------------------------------------------ ingest
// Latents NCHW -> fp32 NHWC; optionally forms z = z_prev + lambda*v_prev first (Algorithm 2,
// hit branch) and writes z and the new motion vector back in the latents' own layout/dtype.
template <typename T>
__global__ void ingest_kernel(IngestArgs a) {
    griddep_launch();
    griddep_wait();
    const int64_t total = (int64_t)a.B * a.C * a.h * a.w;
    const T* z = (const T*)a.z;
    const T* vp = (const T*)a.v_prev;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        // i indexes the NCHW source
        const int x = (int)(i % a.w);
        const int y = (int)((i / a.w) % a.h);
        const int c = (int)((i / ((int64_t)a.w * a.h)) % a.C);
        const int n = (int)(i / ((int64_t)a.w * a.h * a.C));
        float v = ld_f<T>(z, i);
        if (vp) {
            const float zp = v;
            v = fmaf(a.lambda, ld_f<T>(vp, i), zp);
            if (a.z_out) {               // what is decoded is the latent as stored in its own dtype
                st_f<T>((T*)a.z_out, i, v);
                v = ld_f<T>((const T*)a.z_out, i);
            }
            if (a.v_out) st_f<T>((T*)a.v_out, i, v - zp);
        }
        a.x[(((int64_t)n * a.h + y) * a.w + x) * a.C + c] = v;
    }
}

// ------------------------------------------------------------------------------ GroupNorm stats
// One launch.  Every block reduces a run of pixels of one sample to per-group sums of (x - K) and
// (x - K)^2, where K is a reference value per (sample, group) that every block reads from the same
// place (the mean of the group's first four channels at the sample's centre pixel), so the sums
// of different blocks add without correction terms and a large common offset does not cancel.
// A thread owns one 4-channel slot (inside one group, since C/G is a multiple of 4) and walks down
// the pixels.  The block that arrives last for its sample adds the records of all blocks in a
// fixed order and writes scale and shift; the order of every sum is fixed by the sizes alone, so
// the result is bitwise reproducible and independent of the batch a sample is decoded in.
template <typename T> __device__ __forceinline__ void load4(const T* p, float v[4]);
template <> __device__ __forceinline__ void load4<float>(const float* p, float v[4]) {
    const float4 t = *(const float4*)p;
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <> __device__ __forceinline__ void load4<__nv_bfloat16>(const __nv_bfloat16* p, float v[4]) {
    const uint2 t = *(const uint2*)p;
    v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xffff0000u);
    v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xffff0000u);
}

// Streaming loads of the statistics pass: a line it brings in is the first to leave L2 again, so the lines the
// producing kernel has just written stay resident until the pass reaches them.
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
template <typename T> __device__ __forceinline__ void load4_stream(const T* p, float v[4], uint64_t pol);
template <> __device__ __forceinline__ void load4_stream<float>(const float* p, float v[4], uint64_t pol) {
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p), "l"(pol) : "memory");
}
template <> __device__ __forceinline__ void load4_stream<__nv_bfloat16>(const __nv_bfloat16* p, float v[4], uint64_t pol) {
    uint2 t;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;" : "=r"(t.x), "=r"(t.y) : "l"(p), "l"(pol) : "memory");
    v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xffff0000u);
    v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xffff0000u);
}

constexpr int kGnThreads = 512;
constexpr int kGnFinalLoads = (kGnMaxChunks + 15) / 16;   // records a thread of the last block reads in one round (32 groups: 16 slices)

template <typename T, int U>
__global__ void __launch_bounds__(kGnThreads, 2) gn_stats_kernel(GnArgs a, int chunks, int pix_per_chunk) {
    __shared__ float2 sm[kGnThreads];
    __shared__ int s_last;
    griddep_launch();
    const int slots = a.C / 4;                       // 4-channel slots per pixel (<= kGnThreads)
    const int cpg = a.C / a.G;
    const int slot = threadIdx.x % slots;
    // The per-channel offset does not depend on the kernel before this one: it is read while that kernel finishes.
    // off_k: what the offset adds to the group's reference value; off_c: this thread's four channels;
    // off_fin: the same reference term for the group this thread finalises (threads below G, last block only).
    float off_k = 0.f, off_fin = 0.f;
    float4 off_c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.offset) {
        const float4 og = __ldg((const float4*)(a.offset + (slot * 4 / cpg) * cpg));
        off_k = 0.25f * ((og.x + og.y) + (og.z + og.w));
        off_c = __ldg((const float4*)(a.offset + slot * 4));
        if (threadIdx.x < a.G) {
            const float4 of = __ldg((const float4*)(a.offset + threadIdx.x * cpg));
            off_fin = 0.25f * ((of.x + of.y) + (of.z + of.w));
        }
    }
    griddep_wait();
    const int n = blockIdx.y;
    const int chunk = blockIdx.x;
    const int p0 = chunk * pix_per_chunk;
    const int p1 = min(a.P, p0 + pix_per_chunk);
    const T* x = (const T*)a.x + (size_t)n * a.P * a.C;
    const int rows = kGnThreads / slots;             // pixels handled side by side
    const int row = threadIdx.x / slots;

    float s = 0.f, ss = 0.f;
    if (row < rows && p0 + row < p1) {
        float kv[4];
        load4<T>(x + (size_t)(a.P / 2) * a.C + (slot * 4 / cpg) * cpg, kv);
        // a per-channel offset is taken into the reference value: d = (x + off) - k = x - (k - off)
        const float k = 0.25f * ((kv[0] + kv[1]) + (kv[2] + kv[3])) + off_k;
        const float ko[4] = {k - off_c.x, k - off_c.y, k - off_c.z, k - off_c.w};
        int p = p0 + row;
        const uint64_t pol = policy_evict_first();
        for (; p + (U - 1) * rows < p1; p += U * rows) {        // U independent loads in flight
            float u[U][4];
#pragma unroll
            for (int j = 0; j < U; ++j) load4_stream<T>(x + (size_t)(p + j * rows) * a.C + slot * 4, u[j], pol);
#pragma unroll
            for (int j = 0; j < U; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float d = u[j][e] - ko[e];
                    s += d;
                    ss = fmaf(d, d, ss);
                }
        }
        for (; p < p1; p += rows) {
            float v[4];
            load4<T>(x + (size_t)p * a.C + slot * 4, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float d = v[e] - ko[e];
                s += d;
                ss = fmaf(d, d, ss);
            }
        }
    }
    sm[threadIdx.x] = make_float2(s, ss);
    __syncthreads();
    // one thread per group adds its members: rows x (slots of the group), in a fixed order
    if (threadIdx.x < a.G) {
        const int g = threadIdx.x;
        const int spg = cpg / 4;
        float2 acc = make_float2(0.f, 0.f);
        for (int r = 0; r < rows; ++r)
            for (int sl = g * spg; sl < (g + 1) * spg; ++sl) {
                const float2 v = sm[r * slots + sl];
                acc.x += v.x;
                acc.y += v.y;
            }
        ((float2*)a.partial)[((size_t)n * kGnMaxChunks + chunk) * a.G + g] = acc;
    }
    __syncthreads();

    // The block of this sample that finishes last folds the records into scale and shift.
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int prev = atomicAdd(a.counters + n, 1u);
        s_last = (prev == (unsigned int)chunks - 1u) ? 1 : 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // Thread t adds the records k = t / G, t / G + slices, ... of group t % G (a warp reads whole records:
    // coalesced), the slices are added in a fixed order through shared memory, and every thread then writes
    // scale and shift of the channels c = t, t + 512, ...
    const int slices = kGnThreads / a.G;             // >= 1 (checked by the launcher)
    const int g = threadIdx.x % a.G, sl = threadIdx.x / a.G;
    float2 acc = make_float2(0.f, 0.f);
    if (sl < slices) {
        const float2* rec = (const float2*)a.partial + (size_t)n * kGnMaxChunks * a.G + g;
        for (int k0 = sl; k0 < chunks; k0 += kGnFinalLoads * slices) {
            float2 r[kGnFinalLoads];
            // unconditional loads (a record that does not exist re-reads the first and counts as zero), issued
            // back to back before the first use
#pragma unroll
            for (int i = 0; i < kGnFinalLoads; ++i) {
                const int k = k0 + i * slices;
                const float2* q = rec + (size_t)(k < chunks ? k : sl) * a.G;
                asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(r[i].x), "=f"(r[i].y) : "l"(q));
            }
#pragma unroll
            for (int i = 0; i < kGnFinalLoads; ++i) {
                const bool on = k0 + i * slices < chunks;
                acc.x += on ? r[i].x : 0.f;
                acc.y += on ? r[i].y : 0.f;
            }
        }
    }
    __syncthreads();                                 // the block's own use of sm[] above is over
    sm[threadIdx.x] = acc;
    __syncthreads();
    __shared__ float s_mean[kGnThreads], s_rstd[kGnThreads];
    if (threadIdx.x < a.G) {
        float2 t = make_float2(0.f, 0.f);
        for (int q = 0; q < slices; ++q) {
            const float2 v = sm[q * a.G + threadIdx.x];
            t.x += v.x;
            t.y += v.y;
        }
        float kv[4];
        load4<T>(x + (size_t)(a.P / 2) * a.C + threadIdx.x * cpg, kv);
        const float k = 0.25f * ((kv[0] + kv[1]) + (kv[2] + kv[3])) + off_fin;
        const float inv_n = 1.f / ((float)a.P * (float)cpg);
        const float md = t.x * inv_n;
        const float var = fmaxf(fmaf(-md, md, t.y * inv_n), 0.f);
        s_mean[threadIdx.x] = k + md;
        s_rstd[threadIdx.x] = 1.f / sqrtf(var + a.eps);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < a.C; c += kGnThreads) {
        const int gc = c / cpg;
        const float sc = __ldg(a.gamma + c) * s_rstd[gc];
        a.scale[(size_t)n * a.C + c] = sc;
        a.shift[(size_t)n * a.C + c] = __ldg(a.beta + c) - (s_mean[gc] - (a.offset ? __ldg(a.offset + c) : 0.f)) * sc;
    }
    if (threadIdx.x == 0) a.counters[n] = 0u;        // ready for the next launch
}

__device__ __forceinline__ void bulk_load_stream(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, uint64_t pol) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(pol) : "memory");
}

// ---- the pass for handles whose decodes may be of several frames
constexpr int kGnBlocks = 296;                            // two per SM of a 148-SM device (a block waits for no other)
constexpr int kGnStages = 4, kGnStageBytes = 16384;
constexpr unsigned int kGnMine = 0x40000000u;

// What a thread knows and adds up: a 16-byte piece of a pixel (one or two quads of channels) of every `rows`-th pixel.
template <typename T> struct GnSums {
    static constexpr int E = 16 / (int)sizeof(T), Q = E / 4;
    int cpg, quads, ppp, rows, piece, row;               // channels of a group; quads and pieces of a pixel; pixels side by side
    bool on;
    float off_k[Q], off_c[E];                            // what a per-channel offset adds: to the quads' references, to the channels
    float kv[Q][4];                                      // raw reference pixels
    unsigned long long nk[E / 2], s[Q], ss[Q];           // minus the references (the offset taken in); sums by channel parity
    __device__ __forceinline__ void init(const GnArgs& a, int tid) {
        cpg = a.C / a.G; quads = a.C / 4; ppp = a.C / E; rows = kGnThreads / ppp;
        piece = tid % ppp; row = tid / ppp; on = row < rows;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int c = piece * E + q * 4;
            off_k[q] = 0.f;
            off_c[4 * q] = off_c[4 * q + 1] = off_c[4 * q + 2] = off_c[4 * q + 3] = 0.f;
            if (a.offset) {
                const float4 og = __ldg((const float4*)(a.offset + c / cpg * cpg)), oc = __ldg((const float4*)(a.offset + c));
                off_k[q] = 0.25f * ((og.x + og.y) + (og.z + og.w));
                off_c[4 * q] = oc.x; off_c[4 * q + 1] = oc.y; off_c[4 * q + 2] = oc.z; off_c[4 * q + 3] = oc.w;
            }
        }
    }
    __device__ __forceinline__ void load_refs(const GnArgs& a, int n) {
#pragma unroll
        for (int q = 0; q < Q; ++q) load4<T>((const T*)a.x + ((size_t)n * a.P + a.P / 2) * a.C + (piece * E + q * 4) / cpg * cpg, kv[q]);
    }
    __device__ __forceinline__ void start() {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            // d = (x + off) - k = x - (k - off)
            const float k = 0.25f * ((kv[q][0] + kv[q][1]) + (kv[q][2] + kv[q][3])) + off_k[q];
            nk[2 * q] = pack2(off_c[4 * q] - k, off_c[4 * q + 1] - k);
            nk[2 * q + 1] = pack2(off_c[4 * q + 2] - k, off_c[4 * q + 3] - k);
            s[q] = ss[q] = 0ull;
        }
    }
    __device__ __forceinline__ void add(const uint4& r) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            const unsigned long long v = sizeof(T) == 4 ? pack2(__uint_as_float(w[(2 * e) & 3]), __uint_as_float(w[(2 * e + 1) & 3]))
                                                        : pack2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));
            const unsigned long long d = add2(v, nk[e]);
            s[e / 2] = add2(s[e / 2], d);
            ss[e / 2] = fmaf2(d, d, ss[e / 2]);
        }
    }
    __device__ __forceinline__ void put(float2* sm) const {
        if (!on) return;
#pragma unroll
        for (int q = 0; q < Q; ++q) sm[row * quads + piece * Q + q] = make_float2(sum2(s[q]), sum2(ss[q]));
    }
    // A group's members in the block, rows x (quads of the group), added by 2 to 32 neighbouring threads: valid in the first
    // of them, which are the threads with (tid & (lanes - 1)) == 0, group tid / lanes.
    __device__ __forceinline__ float2 group(const float2* sm, int G, int tid, int lanes) const {
        const int g = tid / lanes, qpg = cpg / 4;
        float2 acc = make_float2(0.f, 0.f);
        if (g < G)
            for (int e = tid & (lanes - 1); e < rows * qpg; e += lanes) {
                const int r = (qpg & (qpg - 1)) == 0 ? e >> (__ffs(qpg) - 1) : e / qpg;
                const float2 v = sm[r * quads + g * qpg + (e - r * qpg)];
                acc.x += v.x;
                acc.y += v.y;
            }
        for (int d = lanes >> 1; d > 0; d >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, d);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, d);
        }
        return acc;
    }
};

// Folds sample n's records into scale and shift, by the 512 summing threads: thread t adds the records k = t / G,
// t / G + slices, ... of group t % G (a warp reads whole records: coalesced), the slices are added in a fixed order through
// shared memory, and every thread then writes scale and shift of the channels c = t, t + 512, ...
template <typename T>
__device__ __forceinline__ void gn_fold(const GnArgs& a, int n, int chunks, int tid, float2* sm, float* s_mean, float* s_rstd) {
    constexpr int kLoads = 8;
    const int cpg = a.C / a.G;
    float ref = 0.f;
    if (tid < a.G) {
        float kf[4];
        load4<T>((const T*)a.x + ((size_t)n * a.P + a.P / 2) * a.C + tid * cpg, kf);
        ref = 0.25f * ((kf[0] + kf[1]) + (kf[2] + kf[3]));
        if (a.offset) {
            const float4 of = __ldg((const float4*)(a.offset + tid * cpg));
            ref += 0.25f * ((of.x + of.y) + (of.z + of.w));
        }
    }
    __threadfence();
    const int slices = kGnThreads / a.G;                 // >= 1 (checked by the launcher)
    const int g = tid % a.G, sl = tid / a.G;
    float2 acc = make_float2(0.f, 0.f);
    if (sl < slices) {
        const float2* rec = (const float2*)a.partial + (size_t)n * kGnMaxChunks * a.G + g;
        for (int k0 = sl; k0 < chunks; k0 += kLoads * slices) {
            float2 r[kLoads];
#pragma unroll
            for (int i = 0; i < kLoads; ++i) {               // (a record that does not exist re-reads the first and counts as zero)
                const int k = k0 + i * slices;
                const float2* q = rec + (size_t)(k < chunks ? k : sl) * a.G;
                asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(r[i].x), "=f"(r[i].y) : "l"(q));
            }
#pragma unroll
            for (int i = 0; i < kLoads; ++i) {
                const bool in = k0 + i * slices < chunks;
                acc.x += in ? r[i].x : 0.f;
                acc.y += in ? r[i].y : 0.f;
            }
        }
    }
    sm[tid] = acc;
    named_barrier_sync(1, kGnThreads);
    if (tid < a.G) {
        float2 t = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int q = 0; q < slices; ++q) {
            const float2 v = sm[q * a.G + tid];
            t.x += v.x;
            t.y += v.y;
        }
        const float inv_n = 1.f / ((float)a.P * (float)cpg);
        const float md = t.x * inv_n;
        const float var = fmaxf(fmaf(-md, md, t.y * inv_n), 0.f);
        s_mean[tid] = ref + md;
        s_rstd[tid] = 1.f / sqrtf(var + a.eps);
    }
    named_barrier_sync(1, kGnThreads);
    for (int c = tid; c < a.C; c += kGnThreads) {
        const int gc = c / cpg;
        const float sc = __ldg(a.gamma + c) * s_rstd[gc];
        a.scale[(size_t)n * a.C + c] = sc;
        a.shift[(size_t)n * a.C + c] = __ldg(a.beta + c) - (s_mean[gc] - (a.offset ? __ldg(a.offset + c) : 0.f)) * sc;
    }
    if (tid == 0) a.counters[n] = 0u;                    // ready for the next launch
    named_barrier_sync(1, kGnThreads);                   // (the next fold writes the same shared memory)
}

// Records and references are those of the kernel above.  Its one block per chunk leaves every wave of 296 blocks to fill and drain
// by itself; here the two resident blocks of an SM walk the chunks of all samples, and nothing on the way may empty the pipe:
// bulk copies (a chunk is one run of bytes) keep 128 KB per SM under way while chunks are summed; a warp of its own writes the
// records and arrives (a fence and an atomic take microseconds behind the loads); samples are folded after the last chunk (a
// block that stops to fold falls behind, is last again, and delays every sample after).  Bound by memory where a launch reads a GB
// or more; below, about 10 us (fp32) and 35 us (bf16, whose chunks are half the bytes for the same hand-over) come on top of the
// bytes at 6.7 to 6.9 TB/s: at 354 and 177 MB DRAM is busy 61 and 42 % of the time, issue slots 56 and 66 %.
// Measured, a decode's launches, the kernel above -> this one, us: eight 720x480 frames, fp32 512 channels at 120x180 (354 MB)
// 102 -> 66, 256 at 240x360 146 -> 122, 256 at 480x720 (2.8 GB) 442 -> 430; bf16 512 at 120x180 (177 MB) 81 -> 60, 256 at 240x360
// 105 -> 85, 128 at 480x720 160 -> 138; four 256x256 frames 128 channels 40 -> 33; all statistics of eight frames 2.91 -> 2.54 ms.  A
// single frame's blocks all run at once, and there this kernel's hand-overs cost 1 us more than they save (14 -> 15, 16 -> 17
// in 256x256): handles for one frame keep the other one.
template <typename T>
__global__ void __launch_bounds__(kGnThreads + 64, 2) gn_batch_kernel(GnArgs a, int chunks, int pix_per_chunk, int items) {
    constexpr int S = kGnStages, PPS = kGnStageBytes / (kGnThreads * 16);
    using Sums = GnSums<T>;
    extern __shared__ __align__(128) uint8_t ring[];
    __shared__ float2 sm[kGnThreads * Sums::Q], s_rec[kGnThreads];
    __shared__ float s_mean[kGnThreads], s_rstd[kGnThreads];
    __shared__ uint32_t s_last;                          // bit k: this block's chunk k (below 32) was its sample's last to arrive
    __shared__ int s_more;                               // a later one was (its counter then holds kGnMine + the block)
    __shared__ uint64_t full[S], empty[S];
    __shared__ uint32_t s_abort;
    volatile uint32_t* abort_flag = &s_abort;
    // named barriers: 1 the summing warps; 2 a chunk's sums are there; 3 they have been read; 4 all is recorded
    constexpr int kSums = 2, kRead = 3, kDone = 4, kBoth = kGnThreads + 32;
    griddep_launch();
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int i = 0; i < S; ++i) { mbar_init(smem_u32(&full[i]), 1); mbar_init(smem_u32(&empty[i]), kGnThreads / 32); }
        s_abort = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int rows = kGnThreads / (a.C / Sums::E);
    const size_t pixbytes = (size_t)a.C * sizeof(T);
    const int stage_pix = kGnStageBytes / (rows * (int)pixbytes) * rows;     // whole rounds of the block's rows
    int n = (int)blockIdx.x / chunks, chunk = (int)blockIdx.x - n * chunks, k = 0;
    auto next = [&]() {
        chunk += (int)gridDim.x;
        while (chunk >= chunks) { chunk -= chunks; ++n; }
        ++k;
    };

    if (tid >= kGnThreads + 32) {
        // ------------------------------------------------ loads
        if (tid == kGnThreads + 32) {
            const uint64_t pol = policy_evict_first();
            uint32_t st = 0, ph = 0;
            int issued = 0;
            bool ok = true;
            griddep_wait();
            for (int item = (int)blockIdx.x; item < items && ok; item += (int)gridDim.x, next()) {
                const int p0 = chunk * pix_per_chunk, len = min(a.P, p0 + pix_per_chunk) - p0;
                const char* src = (const char*)a.x + ((size_t)n * a.P + p0) * pixbytes;
                for (int p = 0; p < len; p += stage_pix) {
                    ok = mbar_wait(smem_u32(&empty[st]), ph ^ 1u, abort_flag);
                    if (!ok) break;
                    const uint32_t bytes = (uint32_t)(min(stage_pix, len - p) * (int)pixbytes), bar = smem_u32(&full[st]);
                    mbar_arrive_expect_tx(bar, bytes);
                    bulk_load_stream(smem_u32(ring) + st * kGnStageBytes, src + (size_t)p * pixbytes, bytes, bar, pol);
                    ++issued;
                    if (++st == (uint32_t)S) { st = 0; ph ^= 1u; }
                }
            }
            // everything has landed once it has been summed; if a wait gave up, what is on its way lands first
            for (int i = 0; i < S && ok; ++i) {
                ok = mbar_wait(smem_u32(&empty[st]), ph ^ 1u, abort_flag);
                if (ok && ++st == (uint32_t)S) { st = 0; ph ^= 1u; }
            }
            if (!ok) cc::land_loads(full, S, issued);
        }
        return;
    }
    if (tid >= kGnThreads) {
        // ------------------------------------------------ records and arrivals
        const int lane = tid - kGnThreads;
        griddep_wait();
        int n_before = 0;
        unsigned int arrived = 0, last = 0, more = 0;
        auto look = [&](int j) {                         // the answer to the arrival of chunk j
            if (arrived != (unsigned int)chunks - 1u) return;
            if (j < 32) last |= 1u << j;
            else { a.counters[n_before] = kGnMine + blockIdx.x; more = 1u; }
        };
        for (int item = (int)blockIdx.x; item < items; item += (int)gridDim.x, next()) {
            named_barrier_sync(kSums, kBoth);
            float2* rec = (float2*)a.partial + ((size_t)n * kGnMaxChunks + chunk) * a.G;
            for (int g = lane; g < a.G; g += 32) rec[g] = s_rec[g];
            named_barrier_arrive(kRead, kBoth);
            __threadfence();
            __syncwarp();
            if (lane == 0) {
                if (k > 0) look(k - 1);
                arrived = atomicAdd(a.counters + n, 1u);
            }
            n_before = n;
        }
        if (lane == 0) { look(k - 1); s_last = last; s_more = (int)more; }
        named_barrier_arrive(kDone, kBoth);
        return;
    }

    // ---------------------------------------------------- sums
    Sums sums;
    sums.init(a, tid);                                   // (the offset does not depend on the kernel before this one)
    int lanes = 32;                                      // threads that add up a group
    while (lanes * a.G > kGnThreads) lanes >>= 1;
    const bool even = rows * sums.ppp == kGnThreads && stage_pix * (int)pixbytes == kGnStageBytes;
    const uint32_t slot0 = smem_u32(ring) + (uint32_t)tid * 16u;     // (the row's and the piece's place in a stage)
    griddep_wait();
    sums.load_refs(a, n);
    uint32_t st = 0, ph = 0;
    for (int item = (int)blockIdx.x; item < items; item += (int)gridDim.x, next()) {
        const int len = min(a.P, (chunk + 1) * pix_per_chunk) - chunk * pix_per_chunk;
        const int n_next = (item + (int)gridDim.x) / chunks;         // (another sample: a block has one chunk of each)
        sums.start();
        // the next sample's references, asked for a chunk ahead; from memory two ahead (a load waits behind the stream's)
        if (n_next < a.B) sums.load_refs(a, n_next);
        if (n_next + 1 < a.B && tid * 128 < (int)pixbytes)
            asm volatile("prefetch.global.L2 [%0];" ::"l"((const char*)a.x + ((size_t)(n_next + 1) * a.P + a.P / 2) * pixbytes + tid * 128));
        for (int p = 0; p < len; p += stage_pix) {
            (void)mbar_wait(smem_u32(&full[st]), ph, abort_flag);
            const uint32_t src = slot0 + st * kGnStageBytes;
            if (even && len - p >= stage_pix) {          // a full stage of a width that divides it: no counting
                uint4 w[PPS];
#pragma unroll
                for (int u = 0; u < PPS; ++u) w[u] = lds_u4(src + (uint32_t)(u * kGnThreads * 16));
#pragma unroll
                for (int u = 0; u < PPS; ++u) sums.add(w[u]);
            } else {
                const int cnt = sums.on ? min(stage_pix, len - p) - sums.row : 0;
                for (int r = 0; r < cnt; r += rows) sums.add(lds_u4(src + (uint32_t)(r * sums.ppp) * 16u));
            }
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(smem_u32(&empty[st]));
            if (++st == (uint32_t)S) { st = 0; ph ^= 1u; }
        }
        if (k > 0) named_barrier_sync(kRead, kBoth);     // the sums of the chunk before have been read
        sums.put(sm);
        named_barrier_sync(1, kGnThreads);
        const float2 total = sums.group(sm, a.G, tid, lanes);
        if (tid / lanes < a.G && (tid & (lanes - 1)) == 0) s_rec[tid / lanes] = total;
        named_barrier_arrive(kSums, kBoth);
    }
    named_barrier_sync(kRead, kBoth);
    named_barrier_sync(kDone, kBoth);
    for (uint32_t m = s_last; m != 0u; m &= m - 1u)
        gn_fold<T>(a, ((int)blockIdx.x + (__ffs((int)m) - 1) * (int)gridDim.x) / chunks, chunks, tid, sm, s_mean, s_rstd);
    if (s_more)
        for (int j = 32; j < k; ++j) {
            const int nj = ((int)blockIdx.x + j * (int)gridDim.x) / chunks;
            if (__ldcg(a.counters + nj) == kGnMine + blockIdx.x) gn_fold<T>(a, nj, chunks, tid, sm, s_mean, s_rstd);
        }
    if (tid == 0 && s_abort && a.status && atomicCAS(a.status, 0u, kStatusGnTimeout) == 0u) {
        a.status[1] = blockIdx.x;
        a.status[2] = 0u;
    }
}

// The same statistics for tensors small enough that the passes above are mostly their own latency: a cluster of eight CTAs
// takes 16 channels (one, two or four groups) of one sample, an eighth of its pixels each; the eight sums meet in the first
// CTA's shared memory, and that CTA writes scale and shift: no records in memory, no arrival counter, no second reading
// phase.  Sums are of (x - K) with the reference value K of the pass above.
// The first CTA's shared memory may be written once that CTA runs: every thread arrives on the cluster's barrier at the start
// and waits for the others before the sums are sent, so the wait lies behind the reads.
constexpr int kGnSplit = 8;
template <typename T, int SPG>                       // SPG: four-channel slots per group (1, 2, 4)
__global__ void __cluster_dims__(kGnSplit, 1, 1) __launch_bounds__(1024 / SPG) gn_cluster_kernel(GnArgs a) {
    constexpr int THREADS = 1024 / SPG, NG = 4 / SPG, ROWS = THREADS / 4, U = 8;
    __shared__ float2 s_warp[THREADS / 32][NG], s_all[NG][kGnSplit];
    cc::cluster_arrive();
    griddep_launch();
    const int rank = blockIdx.x % kGnSplit, n = blockIdx.y, lane = threadIdx.x & 31;
    const int slot = threadIdx.x & 3, row = threadIdx.x >> 2, c0 = (int)blockIdx.x / kGnSplit * 16, cg = c0 + slot / SPG * (SPG * 4);
    const int p0 = (int)((long long)a.P * rank / kGnSplit), p1 = (int)((long long)a.P * (rank + 1) / kGnSplit);
    const T* x = (const T*)a.x + (size_t)n * a.P * a.C;
    float off_k = 0.f;
    float4 off_c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.offset) {
        const float4 og = __ldg((const float4*)(a.offset + cg));
        off_k = 0.25f * ((og.x + og.y) + (og.z + og.w));
        off_c = __ldg((const float4*)(a.offset + c0 + slot * 4));
    }
    griddep_wait();
    float kv[4];
    load4<T>(x + (size_t)(a.P / 2) * a.C + cg, kv);
    const T* q = x + (size_t)(p0 + row) * a.C + c0 + slot * 4;
    const size_t step = (size_t)ROWS * a.C;
    float s = 0.f, ss = 0.f, k = 0.f, ko[4] = {0.f, 0.f, 0.f, 0.f};
    bool first = true;
    for (int p = p0 + row; p < p1; p += U * ROWS, q += U * step) {
        float u[U][4];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            u[j][0] = u[j][1] = u[j][2] = u[j][3] = 0.f;
            if (p + j * ROWS < p1) load4<T>(q + j * step, u[j]);
        }
        if (first) {                                 // (its load is in flight together with the first of the others)
            k = 0.25f * ((kv[0] + kv[1]) + (kv[2] + kv[3])) + off_k;
            ko[0] = k - off_c.x; ko[1] = k - off_c.y; ko[2] = k - off_c.z; ko[3] = k - off_c.w;
            first = false;
        }
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (p + j * ROWS < p1)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float d = u[j][e] - ko[e];
                    s += d;
                    ss = fmaf(d, d, ss);
                }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        if (d >= 4 || d < SPG) {                     // (lane bits 0 and 1 are the slot)
            s += __shfl_xor_sync(0xffffffffu, s, d);
            ss += __shfl_xor_sync(0xffffffffu, ss, d);
        }
    }
    if (lane < 4 && lane % SPG == 0) s_warp[threadIdx.x / 32][lane / SPG] = make_float2(s, ss);
    __syncthreads();
    cc::cluster_wait();                              // every CTA of the cluster runs
    if (threadIdx.x < NG) {
        float2 t = s_warp[0][threadIdx.x];
#pragma unroll 8
        for (int w = 1; w < THREADS / 32; ++w) { t.x += s_warp[w][threadIdx.x].x; t.y += s_warp[w][threadIdx.x].y; }
        const uint32_t dst = tc::map_to_cta(tc::smem_u32(&s_all[threadIdx.x][rank]), 0u);
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(t.x), "f"(t.y) : "memory");
    }
    __syncwarp();
    cc::cluster_arrive();
    cc::cluster_wait();                              // the sums have arrived
    if (rank != 0 || threadIdx.x >= 16) return;
    const int g = threadIdx.x / (SPG * 4), c = c0 + threadIdx.x;
    float2 t = s_all[g][0];
#pragma unroll
    for (int r = 1; r < kGnSplit; ++r) { t.x += s_all[g][r].x; t.y += s_all[g][r].y; }
    load4<T>(x + (size_t)(a.P / 2) * a.C + c0 + g * SPG * 4, kv);
    float kk = 0.25f * ((kv[0] + kv[1]) + (kv[2] + kv[3]));
    if (a.offset) {
        const float4 og = __ldg((const float4*)(a.offset + c0 + g * SPG * 4));
        kk += 0.25f * ((og.x + og.y) + (og.z + og.w));
    }
    const float inv_n = 1.f / ((float)a.P * (float)(SPG * 4));
    const float md = t.x * inv_n, var = fmaxf(fmaf(-md, md, t.y * inv_n), 0.f);
    const float sc = __ldg(a.gamma + c) * (1.f / sqrtf(var + a.eps));
    a.scale[(size_t)n * a.C + c] = sc;
    a.shift[(size_t)n * a.C + c] = __ldg(a.beta + c) - (kk + md - (a.offset ? __ldg(a.offset + c) : 0.f)) * sc;
}

// ------------------------------------------------------------------------------- direct conv
// Block = TH x TW output pixels x CT output channels; input channels are consumed KC at a time
// through shared memory (the transformed input tile with its halo, and the weight slice).
constexpr int KC = 8;

template <typename TIn, typename TOut, int TH, int TW, int PPT, int CPT, int CGROUPS>
__global__ void __launch_bounds__((TH * TW / PPT) * CGROUPS) conv_simt_kernel(ConvArgs a) {
    griddep_launch();
    griddep_wait();
    constexpr int NPG = TH * TW / PPT;
    constexpr int CT = CPT * CGROUPS;
    constexpr int NT = NPG * CGROUPS;
    constexpr int PW = TW + 2, PH = TH + 2, NPIX = PW * PH;
    __shared__ float s_in[KC][NPIX + 1];
    __shared__ float s_w[9][KC][CT];

    const int tiles_x = (a.W + TW - 1) / TW;
    const int tx0 = (blockIdx.x % tiles_x) * TW;
    const int ty0 = (blockIdx.x / tiles_x) * TH;
    const int ct0 = blockIdx.y * CT;
    const int b = blockIdx.z;
    const int tid = threadIdx.x;
    const int pg = tid % NPG, cg = tid / NPG;
    const int ly = (pg * PPT) / TW, lx = (pg * PPT) % TW;
    const int taps = a.ksize * a.ksize;
    const int up = a.upsample ? 1 : 0;

    float acc[PPT][CPT];
#pragma unroll
    for (int p = 0; p < PPT; ++p)
#pragma unroll
        for (int q = 0; q < CPT; ++q) acc[p][q] = 0.f;

    const TIn* x = (const TIn*)a.x + (size_t)b * a.Hs * a.Ws * a.Cin;
    const float* wp = (const float*)a.w;

    for (int c0 = 0; c0 < a.Cin; c0 += KC) {
        for (int idx = tid; idx < NPIX * KC; idx += NT) {
            const int c = idx % KC, pix = idx / KC;
            const int oy = ty0 + pix / PW - 1, ox = tx0 + pix % PW - 1;
            float v = 0.f;
            if (oy >= 0 && oy < a.H && ox >= 0 && ox < a.W && c0 + c < a.Cin) {
                v = ld_f<TIn>(x, ((size_t)(oy >> up) * a.Ws + (ox >> up)) * a.Cin + c0 + c);
                if (a.scale) v = fmaf(v, a.scale[(size_t)b * a.Cin + c0 + c], a.shift[(size_t)b * a.Cin + c0 + c]);
                if (a.silu) v = silu_f(v);
                if (a.bf16_operands) v = round_bf16(v);
            }
            s_in[c][pix] = v;
        }
        for (int idx = tid; idx < taps * KC * CT; idx += NT) {
            const int ct = idx % CT, c = (idx / CT) % KC, tap = idx / (CT * KC);
            float v = 0.f;
            if (c0 + c < a.Cin && ct0 + ct < a.Cout) v = wp[((size_t)tap * a.Cin + c0 + c) * a.Cout + ct0 + ct];
            s_w[tap][c][ct] = v;
        }
        __syncthreads();
        for (int tap = 0; tap < taps; ++tap) {
            const int dy = a.ksize == 3 ? tap / 3 : 1, dx = a.ksize == 3 ? tap % 3 : 1;
            const int base = (ly + dy) * PW + lx + dx;
#pragma unroll
            for (int c = 0; c < KC; ++c) {
                float iv[PPT], wv[CPT];
#pragma unroll
                for (int p = 0; p < PPT; ++p) iv[p] = s_in[c][base + p];
#pragma unroll
                for (int q = 0; q < CPT; ++q) wv[q] = s_w[tap][c][cg * CPT + q];
#pragma unroll
                for (int p = 0; p < PPT; ++p)
#pragma unroll
                    for (int q = 0; q < CPT; ++q) acc[p][q] = fmaf(iv[p], wv[q], acc[p][q]);
            }
        }
        __syncthreads();
    }

    TOut* y = (TOut*)a.y;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        const int oy = ty0 + ly, ox = tx0 + lx + p;
        if (oy >= a.H || ox >= a.W) continue;
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int co = ct0 + cg * CPT + q;
            if (co >= a.Cout) continue;
            float v = acc[p][q];
            if (a.bias) v += a.bias[co];
            const size_t nhwc = (((size_t)b * a.H + oy) * a.W + ox) * a.Cout + co;
            if (a.residual) v += a.residual[nhwc];
            const size_t o = a.out_nchw ? (((size_t)b * a.Cout + co) * a.H + oy) * a.W + ox : nhwc;
            if (a.out_u8) ((unsigned char*)a.y)[nhwc] = pack_u8(v);
            else st_f<TOut>(y, o, v);
        }
    }
}

template <typename TIn, typename TOut>
cudaError_t conv_simt_dispatch(const ConvArgs& a, cudaStream_t s) {
    if (a.Cout <= 8) {
        constexpr int TH = 16, TW = 16, CT = 4;
        dim3 grid(((a.W + TW - 1) / TW) * ((a.H + TH - 1) / TH), (a.Cout + CT - 1) / CT, a.B);
        launch_pdl(conv_simt_kernel<TIn, TOut, TH, TW, 1, 4, 1>, grid, dim3(256), 0, s, a);
    } else {
        constexpr int TH = 8, TW = 8, CT = 64;
        dim3 grid(((a.W + TW - 1) / TW) * ((a.H + TH - 1) / TH), (a.Cout + CT - 1) / CT, a.B);
        launch_pdl(conv_simt_kernel<TIn, TOut, TH, TW, 4, 4, 16>, grid, dim3(256), 0, s, a);
    }
    return cudaGetLastError();
}

// --------------------------------------------------------------------------------- attention
// Softmax attention in fp32 on the FP32 pipes, for the few tokens of the mid block of small frames (64 for a 64x64 frame)
// in the single-precision path.  A CTA of eight warps takes QT queries and walks 64 keys at a time with a running maximum and
// sum.  Scores: a warp has eight keys; a lane takes four channels of every 128 and keeps all 8 x QT partial sums, which one
// halving exchange over the warp adds up (31 shuffles instead of 5 per sum).  Output: a thread has four channels and every
// second key.  K and V go straight from L2 to registers: no key is used twice by a thread, and staging
// them cost more than the products (one warp per query, 8 queries per CTA: 8 CTAs at 64 tokens, 76 us; now 12).
// QT = 2 as long as the CTAs fit the chip at once, 4 beyond (K and V are read T / QT times).
constexpr int kAttnTile = 64, kAttnMaxC = 512;

__device__ __forceinline__ float4 attn_ld4(const float* p, bool vec) {
    return vec ? __ldcg((const float4*)p) : make_float4(p[0], p[1], p[2], p[3]);
}

// Sums of v[0..N) over the warp: v[0] of lane i is the sum of value i / (32 / N).
template <int N> __device__ __forceinline__ void warp_sums(float (&v)[N], int lane) {
#pragma unroll
    for (int d = 16, n = N; d > 0; d >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = lane & d;
#pragma unroll
            for (int i = 0; i < N / 2; ++i)
                if (i < n) {
                    const float other = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + n], d);
                    v[i] = (up ? v[i + n] : v[i]) + other;
                }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
        }
    }
}

template <int QT>
__global__ void __launch_bounds__(256, 2) attn_f32_kernel(AttnArgs a, bool vec) {
    __shared__ __align__(16) float s_q[QT][kAttnMaxC];
    __shared__ __align__(16) float s_p[kAttnTile * QT];      // [key][query]
    __shared__ float s_corr[QT], s_l[QT];
    __shared__ float4 s_o[QT][kAttnMaxC / 4];
    griddep_launch();
    griddep_wait();
    const int C = a.C, b = blockIdx.y, q0 = blockIdx.x * QT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, half = tid >> 7, c4 = (tid & 127) * 4;
    const float* q = (const float*)a.q + (size_t)b * a.T * a.ld_qkv;
    const float* k = (const float*)a.k + (size_t)b * a.T * a.ld_qkv;
    const float* v = (const float*)a.v + (size_t)b * a.T * a.ld_qkv;
    for (int i = tid; i < QT * (kAttnMaxC / 4); i += 256) {
        const int t = i / (kAttnMaxC / 4), c = i % (kAttnMaxC / 4) * 4;
        *(float4*)&s_q[t][c] = q0 + t < a.T && c < C ? attn_ld4(q + (size_t)(q0 + t) * a.ld_qkv + c, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float4 acc[QT];
#pragma unroll
    for (int t = 0; t < QT; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    float m = -INFINITY, l = 0.f;                            // of query `warp` (warps 0..QT-1)
    __syncthreads();
#pragma unroll 1
    for (int k0 = 0; k0 < a.T; k0 += kAttnTile) {
        float sc[8 * QT];
#pragma unroll
        for (int i = 0; i < 8 * QT; ++i) sc[i] = 0.f;
#pragma unroll
        for (int i = 0; i < kAttnMaxC / 128; ++i) {
            const int c = i * 128 + lane * 4;
            float4 kv[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int key = k0 + warp * 8 + e;
                kv[e] = c < C && key < a.T ? attn_ld4(k + (size_t)key * a.ld_qkv + c, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int t = 0; t < QT; ++t) {
                const float4 qv = *(const float4*)&s_q[t][c];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    sc[e * QT + t] = fmaf(qv.w, kv[e].w, fmaf(qv.z, kv[e].z, fmaf(qv.y, kv[e].y, fmaf(qv.x, kv[e].x, sc[e * QT + t]))));
            }
        }
        warp_sums<8 * QT>(sc, lane);
        if (lane % (4 / QT) == 0) {
            const int i = lane / (4 / QT);
            s_p[warp * 8 * QT + i] = k0 + warp * 8 + i / QT < a.T ? sc[0] * a.scale : -INFINITY;
        }
        __syncthreads();
        if (warp < QT) {
            const float x0 = s_p[lane * QT + warp], x1 = s_p[(lane + 32) * QT + warp];
            float top = fmaxf(x0, x1);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
            const float m_new = fmaxf(m, top);               // finite: every tile has a key
            const float corr = expf(m - m_new), p0 = expf(x0 - m_new), p1 = expf(x1 - m_new);
            float sum = p0 + p1;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
            l = l * corr + sum;
            m = m_new;
            s_p[lane * QT + warp] = p0;
            s_p[(lane + 32) * QT + warp] = p1;
            if (lane == 0) { s_corr[warp] = corr; s_l[warp] = l; }
        }
        __syncthreads();
        if (c4 < C) {
#pragma unroll
            for (int t = 0; t < QT; ++t) {
                const float corr = s_corr[t];
                acc[t].x *= corr; acc[t].y *= corr; acc[t].z *= corr; acc[t].w *= corr;
            }
            constexpr int U = 16;                            // keys on their way at a time
#pragma unroll 1
            for (int e0 = half; e0 < kAttnTile && k0 + e0 < a.T; e0 += 2 * U) {
                float4 vv[U];
#pragma unroll
                for (int e = 0; e < U; ++e)
                    vv[e] = k0 + e0 + 2 * e < a.T ? attn_ld4(v + (size_t)(k0 + e0 + 2 * e) * a.ld_qkv + c4, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int e = 0; e < U; ++e)
#pragma unroll
                    for (int t = 0; t < QT; ++t) {
                        const float p = s_p[(e0 + 2 * e) * QT + t];
                        acc[t].x = fmaf(p, vv[e].x, acc[t].x); acc[t].y = fmaf(p, vv[e].y, acc[t].y);
                        acc[t].z = fmaf(p, vv[e].z, acc[t].z); acc[t].w = fmaf(p, vv[e].w, acc[t].w);
                    }
            }
        }
        __syncthreads();
    }
    if (half == 1 && c4 < C) {
#pragma unroll
        for (int t = 0; t < QT; ++t) s_o[t][c4 / 4] = acc[t];
    }
    __syncthreads();
    if (half == 0 && c4 < C) {
        float* o = (float*)a.o + ((size_t)b * a.T + q0) * a.ld_o + c4;
#pragma unroll
        for (int t = 0; t < QT; ++t) {
            if (q0 + t >= a.T) break;
            const float inv = 1.f / s_l[t];
            const float4 r = s_o[t][c4 / 4];
            float* d = o + (size_t)t * a.ld_o;
            d[0] = (acc[t].x + r.x) * inv; d[1] = (acc[t].y + r.y) * inv; d[2] = (acc[t].z + r.z) * inv; d[3] = (acc[t].w + r.w) * inv;
        }
    }
}

// bf16 tensors, which take this path only where the FFMA kernels are asked for as a check: one warp per query, eight queries
// per block sharing 32-key K/V tiles in shared memory; running maximum / running sum softmax, all in fp32.
constexpr int kAttnQ = 8, kAttnKeys = 32;

__global__ void __launch_bounds__(kAttnQ * 32) attn_bf16_kernel(AttnArgs a) {
    using T = __nv_bfloat16;
    griddep_launch();
    griddep_wait();
    extern __shared__ float smem[];
    const int C = a.C;
    float* s_q = smem;                               // [kAttnQ][C]
    float* s_k = s_q + kAttnQ * C;                   // [kAttnKeys][C+1]
    float* s_v = s_k + kAttnKeys * (C + 1);          // [kAttnKeys][C]
    const int b = blockIdx.y;
    const int q0 = blockIdx.x * kAttnQ;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const T* q = (const T*)a.q + (size_t)b * a.T * a.ld_qkv;
    const T* k = (const T*)a.k + (size_t)b * a.T * a.ld_qkv;
    const T* v = (const T*)a.v + (size_t)b * a.T * a.ld_qkv;
    T* o = (T*)a.o + (size_t)b * a.T * a.ld_o;

    for (int idx = threadIdx.x; idx < kAttnQ * C; idx += blockDim.x) {
        const int qi = idx / C, c = idx % C;
        s_q[idx] = (q0 + qi < a.T) ? ld_f<T>(q, (size_t)(q0 + qi) * a.ld_qkv + c) : 0.f;
    }
    const int nacc = C / 32;                          // channels per lane (C multiple of 32, <= 512)
    float acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.f;
    float m = -INFINITY, l = 0.f;

    for (int k0 = 0; k0 < a.T; k0 += kAttnKeys) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < kAttnKeys * C; idx += blockDim.x) {
            const int ki = idx / C, c = idx % C;
            const bool ok = k0 + ki < a.T;
            s_k[ki * (C + 1) + c] = ok ? ld_f<T>(k, (size_t)(k0 + ki) * a.ld_qkv + c) : 0.f;
            s_v[ki * C + c] = ok ? ld_f<T>(v, (size_t)(k0 + ki) * a.ld_qkv + c) : 0.f;
        }
        __syncthreads();
        float sc = 0.f;
        const float* qr = s_q + warp * C;
        const float* kr = s_k + lane * (C + 1);
        for (int c = 0; c < C; ++c) sc = fmaf(qr[c], kr[c], sc);
        sc = (k0 + lane < a.T) ? sc * a.scale : -INFINITY;
        float tmax = sc;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, d));
        const float m_new = fmaxf(m, tmax);
        const float corr = expf(m - m_new);           // m = -inf at the first tile: exp(-inf) = 0
        const float p = expf(sc - m_new);
        float psum = p;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, d);
        l = l * corr + psum;
        m = m_new;
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] *= corr;
        for (int ki = 0; ki < kAttnKeys; ++ki) {
            const float pk = __shfl_sync(0xffffffffu, p, ki);
            const float* vr = s_v + ki * C + lane;
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (i < nacc) acc[i] = fmaf(pk, vr[i * 32], acc[i]);
        }
    }
    if (q0 + warp < a.T) {
        const float inv = 1.f / l;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < nacc) st_f<T>(o, (size_t)(q0 + warp) * a.ld_o + lane + i * 32, acc[i] * inv);
    }
}

// ------------------------------------------------------------------------------------ repack
template <typename T>
__global__ void pack_weight_simt_kernel(const T* w, float* packed, int Cout, int Cin, int taps, int cout_total,
                                        int cout_offset) {
    const int64_t total = (int64_t)Cout * Cin * taps;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int tap = (int)(i % taps);
        const int c = (int)((i / taps) % Cin);
        const int o = (int)(i / ((int64_t)taps * Cin));
        packed[((size_t)tap * Cin + c) * cout_total + cout_offset + o] = ld_f<T>(w, i);
    }
}

template <typename T>
__global__ void to_f32_kernel(const T* src, float* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = ld_f<T>(src, i);
}

int grid_for(int64_t n, int threads) {
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 148 * 16) g = 148 * 16;
    return (int)g;
}

}  // namespace

cudaError_t launch_ingest(const IngestArgs& a, cudaStream_t s) {
    const int64_t n = (int64_t)a.B * a.C * a.h * a.w;
    if (a.dtype == VD_BF16) launch_pdl(ingest_kernel<__nv_bfloat16>, dim3(grid_for(n, 256)), dim3(256), 0, s, a);
    else launch_pdl(ingest_kernel<float>, dim3(grid_for(n, 256)), dim3(256), 0, s, a);
    return cudaGetLastError();
}

bool gn_takes_clusters(const GnArgs& a) {
    const int spg = a.C / a.G / 4;
    // Up to here the clusters' few CTAs read a sample faster than the other kernel's phases run (the line depends on the
    // sample size only, like everything below).  Measured by itself, one sample, us, other kernel -> this one, a 2 us memset
    // included in both: 512 channels 32x32 10.3 -> 6.3, 60x90 10.4 -> 8.2; 256 channels 128x128 12.2 -> 8.6, bf16 240x360
    // 14.5 -> 20.7; 128 channels 296x424 14.5 -> 16.5.  The line is that of whole decodes, where the other kernel's pass leaves
    // the next layer's lines in L2: 424x296 1565 -> 1536 us with it at 3 million elements, 1567 at 12 million, 1666 at 20 million;
    // from 3 to 4.5 million (256 channels at 128x128 then come here) 256x256 957 -> 962, 288x224 1062 -> 1067, 320x192
    // 1007 -> 1013, 424x296 1470 -> 1472, four 256x256 frames 2648 -> 2634.
    return !a.no_clusters && a.C % 16 == 0 && (spg == 1 || spg == 2 || spg == 4) && (long long)a.P * a.C <= 3000000;
}

bool gn_clusters_fit() {
    return cc::clusters_fit<gn_cluster_kernel<float, 1>>(1024, 0, kGnSplit) && cc::clusters_fit<gn_cluster_kernel<__nv_bfloat16, 1>>(1024, 0, kGnSplit);
}

namespace {
template <typename T>
cudaError_t launch_gn_batch(const GnArgs& a, int chunks, int ppc, cudaStream_t s) {
    constexpr int SMEM = kGnStages * kGnStageBytes;
    const cudaError_t e = cc::set_smem_limit<gn_batch_kernel<T>>(SMEM);
    if (e != cudaSuccess) return e;
    const int items = chunks * a.B;
    return launch_pdl(gn_batch_kernel<T>, dim3(min(items, kGnBlocks)), dim3(kGnThreads + 64), SMEM, s, a, chunks, ppc, items);
}
}  // namespace

cudaError_t launch_gn_stats(const GnArgs& a, cudaStream_t s) {
    if (a.C % 4 != 0 || a.C / 4 > kGnThreads || a.G > kGnThreads || (a.C / a.G) % 4 != 0) return cudaErrorInvalidValue;
    if (gn_takes_clusters(a) && gn_clusters_fit()) {
        const int spg = a.C / a.G / 4;
        const dim3 grid(a.C / 16 * kGnSplit, a.B), block(1024 / spg);
        if (a.dtype == VD_BF16)
            return spg == 4 ? launch_pdl(gn_cluster_kernel<__nv_bfloat16, 4>, grid, block, 0, s, a)
                 : spg == 2 ? launch_pdl(gn_cluster_kernel<__nv_bfloat16, 2>, grid, block, 0, s, a) : launch_pdl(gn_cluster_kernel<__nv_bfloat16, 1>, grid, block, 0, s, a);
        return spg == 4 ? launch_pdl(gn_cluster_kernel<float, 4>, grid, block, 0, s, a)
             : spg == 2 ? launch_pdl(gn_cluster_kernel<float, 2>, grid, block, 0, s, a) : launch_pdl(gn_cluster_kernel<float, 1>, grid, block, 0, s, a);
    }
    // chunks per sample depend on the sample size only (so a frame's statistics, and with them
    // the frame, do not depend on the batch it is decoded in): at least 32 (16) pixels per chunk
    if (!a.single && aligned16(a.x) && (a.dtype != VD_BF16 || a.C % 8 == 0)) {       // (every pixel is whole 16-byte pieces)
        if (a.B < 1 || a.B > 65535) return cudaErrorInvalidConfiguration;
        const int ppc = max(16, (a.P + kGnMaxChunks - 1) / kGnMaxChunks), chunks = (a.P + ppc - 1) / ppc;
        return a.dtype == VD_BF16 ? launch_gn_batch<__nv_bfloat16>(a, chunks, ppc, s) : launch_gn_batch<float>(a, chunks, ppc, s);
    }
    int ppc = max(32, (a.P + kGnMaxChunks - 1) / kGnMaxChunks);
    int chunks = (a.P + ppc - 1) / ppc;
    dim3 grid(chunks, a.B);
    if (a.dtype == VD_BF16) launch_pdl(gn_stats_kernel<__nv_bfloat16, 16>, grid, dim3(kGnThreads), 0, s, a, chunks, ppc);
    else launch_pdl(gn_stats_kernel<float, 8>, grid, dim3(kGnThreads), 0, s, a, chunks, ppc);
    return cudaGetLastError();
}

// The first convolution (latent channels -> hundreds of channels): K = 9 * Cin <= 72 is too thin for the tensor core and for
// the staging of the tiled FFMA kernels.  A block computes 64 (32, 16) consecutive pixels of a frame x 128 output channels; a
// thread holds 8 (4, 2) pixels x 4 channels.  The weights go to shared memory while the kernel before is still running, the
// pixels' 3x3 neighbourhoods as float4 of channels after it: per four k's and thread 4 + 8 shared loads of 16 bytes for 128
// multiply-adds, and these loads are the bound (three blocks per SM, or blocks that walk the image with the weights in place,
// are no faster).  The output's GroupNorm statistics leave as records (conv_cluster.cuh).  4->512, profiled, the tiled
// kernel -> this one: 37x53 17 -> 12 us, 60x90 30 -> 21, two 90x160 frames 119 -> 57.
constexpr int kThinCout = 128, kThinWarps = 8;
// pixels of a thread: two where that gives small images more blocks (and few enough records for the next layer to merge
// itself); else as many as shared memory has room for
static int thin_px(const ConvArgs& a) { return a.H * a.W <= 256 ? 2 : a.Cin == 4 ? 8 : 4; }
template <int CIN, int PX>
__global__ void __launch_bounds__(256, 2) conv_thin_kernel(ConvArgs a) {
    constexpr int K = 9 * CIN, K4 = K / 4, PIX = PX * kThinWarps;
    __shared__ float4 s_x[K4][PIX];
    __shared__ float4 s_w[K][kThinCout / 4];
    griddep_launch();
    const int P = a.H * a.W, blocks = (P + PIX - 1) / PIX;
    const int frame = blockIdx.x / blocks, block = blockIdx.x - frame * blocks, p0 = block * PIX;
    const int co0 = blockIdx.y * kThinCout, tid = threadIdx.x, pg = tid >> 5, cg = tid & 31, co = co0 + cg * 4;
    for (int i = tid; i < K * (kThinCout / 4); i += 256) {
        const int k = i / (kThinCout / 4), c = i % (kThinCout / 4);
        s_w[k][c] = __ldg((const float4*)((const float*)a.w + (size_t)k * a.Cout + co0) + c);
    }
    float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.bias) bias = __ldg((const float4*)(a.bias + co));
    const int px = p0 + (tid & (PIX - 1)), oy = px / a.W, ox = px - oy * a.W;        // this thread's pixel of the gather
    const float4* x = (const float4*)a.x + (size_t)frame * P * (CIN / 4);
    griddep_wait();
#pragma unroll
    for (int r = tid / PIX; r < K4; r += 256 / PIX) {
        const int tap = r / (CIN / 4), yy = oy + tap / 3 - 1, xx = ox + tap % 3 - 1;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (px < P && yy >= 0 && yy < a.H && xx >= 0 && xx < a.W) v = __ldcg(x + ((size_t)yy * a.W + xx) * (CIN / 4) + r % (CIN / 4));
        if (a.bf16_operands) v = make_float4(round_bf16(v.x), round_bf16(v.y), round_bf16(v.z), round_bf16(v.w));
        s_x[r][tid & (PIX - 1)] = v;
    }
    __syncthreads();
    float acc[PX][4];
#pragma unroll
    for (int i = 0; i < PX; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = 0.f;
#pragma unroll 3
    for (int k4 = 0; k4 < K4; ++k4) {
        float4 xv[PX];
#pragma unroll
        for (int i = 0; i < PX; ++i) xv[i] = s_x[k4][pg * PX + i];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float4 w = s_w[k4 * 4 + e][cg];
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                const float v = e == 0 ? xv[i].x : e == 1 ? xv[i].y : e == 2 ? xv[i].z : xv[i].w;
                acc[i][0] = fmaf(v, w.x, acc[i][0]); acc[i][1] = fmaf(v, w.y, acc[i][1]);
                acc[i][2] = fmaf(v, w.z, acc[i][2]); acc[i][3] = fmaf(v, w.w, acc[i][3]);
            }
        }
    }
    const int n = min(max(P - p0 - pg * PX, 0), PX);         // pixels of this warp
    float* y = (float*)a.y + ((size_t)frame * P + p0 + pg * PX) * a.Cout + co;
    float sum = 0.f, sq = 0.f, pivot = 0.f;
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        const float4 v = make_float4(acc[i][0] + bias.x, acc[i][1] + bias.y, acc[i][2] + bias.z, acc[i][3] + bias.w);
        if (i < n) *(float4*)(y + (size_t)i * a.Cout) = v;
        if (a.out_rec) {                                     // a group is 1 << (out_shift - 2) lanes
            if (i == 0) pivot = __shfl_sync(0xffffffffu, v.x, cg & ~((1 << (a.out_shift - 2)) - 1));
            if (i < n) {
                const float d0 = v.x - pivot, d1 = v.y - pivot, d2 = v.z - pivot, d3 = v.w - pivot;
                sum += (d0 + d1) + (d2 + d3);
                sq += fmaf(d0, d0, d1 * d1) + fmaf(d2, d2, d3 * d3);
            }
        }
    }
    if (a.out_rec) {
#pragma unroll
        for (int d = 1; d < 4; d <<= 1)
            if (d < 1 << (a.out_shift - 2)) {
                sum += __shfl_xor_sync(0xffffffffu, sum, d);
                sq += __shfl_xor_sync(0xffffffffu, sq, d);
            }
        if ((cg & ((1 << (a.out_shift - 2)) - 1)) == 0) {
            const float cnt = (float)(n << a.out_shift), dm = n ? sum / cnt : 0.f;
            a.out_rec[((size_t)frame * a.out_G + (co >> a.out_shift)) * a.out_slots + block * kThinWarps + pg] =
                make_float4(cnt, pivot + dm, fmaxf(fmaf(-dm, sum, sq), 0.f), 0.f);
        }
    }
}

bool conv_thin_supported(const ConvArgs& a) {
    return a.in_dtype == VD_F32 && a.out_dtype == VD_F32 && a.ksize == 3 && (a.Cin == 4 || a.Cin == 8) && a.Cout % kThinCout == 0 && !a.scale && !a.silu &&
           !a.residual && !a.upsample && !a.out_nchw && !a.out_u8 && !a.x2 &&
           aligned16(a.x) && aligned16(a.w) && aligned16(a.bias) && aligned16(a.y);      // all read and written as float4
}
int conv_thin_slots(const ConvArgs& a) { return (a.H * a.W + thin_px(a) * kThinWarps - 1) / (thin_px(a) * kThinWarps) * kThinWarps; }

cudaError_t launch_conv_simt(const ConvArgs& a, cudaStream_t s) {
    const bool ib = a.in_dtype == VD_BF16, ob = a.out_dtype == VD_BF16;
    if (a.upsample == 2) return cudaErrorInvalidValue;       // its weights are packed as sixteen 2x2 taps, which these kernels do not read
    if (conv_thin_supported(a)) {
        if (a.out_rec && !rec_groups_ok(a.Cout, a.out_G)) return cudaErrorInvalidValue;
        const long long blocks = (long long)conv_thin_slots(a) / kThinWarps * a.B;
        if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
        const dim3 grid((unsigned)blocks, a.Cout / kThinCout);
        auto launch = [&](auto kern) { return launch_pdl(kern, grid, dim3(256), 0, s, a); };
        if (thin_px(a) == 2) return a.Cin == 4 ? launch(conv_thin_kernel<4, 2>) : launch(conv_thin_kernel<8, 2>);
        return a.Cin == 4 ? launch(conv_thin_kernel<4, 8>) : launch(conv_thin_kernel<8, 4>);
    }
    if (ib && ob) return conv_simt_dispatch<__nv_bfloat16, __nv_bfloat16>(a, s);
    if (ib && !ob) return conv_simt_dispatch<__nv_bfloat16, float>(a, s);
    if (!ib && ob) return conv_simt_dispatch<float, __nv_bfloat16>(a, s);
    return conv_simt_dispatch<float, float>(a, s);
}

cudaError_t launch_attn_simt(const AttnArgs& a, cudaStream_t s) {
    if (a.C % 32 != 0 || a.C > 512) return cudaErrorInvalidValue;
    if (a.dtype == VD_BF16) {
        const size_t smem = sizeof(float) * ((size_t)kAttnQ * a.C + (size_t)kAttnKeys * (a.C + 1) + (size_t)kAttnKeys * a.C);
        const cudaError_t e = cudaFuncSetAttribute(attn_bf16_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        launch_pdl(attn_bf16_kernel, dim3((a.T + kAttnQ - 1) / kAttnQ, a.B), dim3(kAttnQ * 32), smem, s, a);
        return cudaGetLastError();
    }
    const bool vec = a.ld_qkv % 4 == 0 && (((uintptr_t)a.q | (uintptr_t)a.k | (uintptr_t)a.v) & 15) == 0;
    const int qt = (long long)a.B * ((a.T + 1) / 2) <= 2 * 148 ? 2 : 4;
    const dim3 grid((a.T + qt - 1) / qt, a.B);
    if (qt == 2) launch_pdl(attn_f32_kernel<2>, grid, dim3(256), 0, s, a, vec);
    else launch_pdl(attn_f32_kernel<4>, grid, dim3(256), 0, s, a, vec);
    return cudaGetLastError();
}

cudaError_t launch_pack_weight_simt(const void* w, int w_dtype, float* packed, int Cout, int Cin, int taps,
                                    int cout_total, int cout_offset, cudaStream_t s) {
    const int64_t n = (int64_t)Cout * Cin * taps;
    if (w_dtype == VD_BF16)
        pack_weight_simt_kernel<__nv_bfloat16><<<grid_for(n, 256), 256, 0, s>>>((const __nv_bfloat16*)w, packed, Cout, Cin, taps, cout_total, cout_offset);
    else
        pack_weight_simt_kernel<float><<<grid_for(n, 256), 256, 0, s>>>((const float*)w, packed, Cout, Cin, taps, cout_total, cout_offset);
    return cudaGetLastError();
}

__global__ void fold_bias_kernel(float* out, const float* in, const float* b, const float* b2, const float* w2, const float* pin,
                                 int Cin2, int Cout) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= Cout) return;
    float v = (in ? in[c] : 0.f) + (b ? b[c] : 0.f) + (b2 ? b2[c] : 0.f);
    if (w2 && pin) {
        float acc = 0.f;
        for (int k = 0; k < Cin2; ++k) acc = fmaf(w2[(size_t)c * Cin2 + k], pin[k], acc);
        v += acc;
    }
    out[c] = v;
}
__global__ void fill_rows_kernel(float* dst, const float* src, int C, int B) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < C * B) dst[i] = src ? src[i % C] : 1.f;
}
cudaError_t launch_fold_bias(float* out, const float* in, const float* b, const float* b2, const float* w2, const float* pin,
                             int Cin2, int Cout, cudaStream_t s) {
    fold_bias_kernel<<<(Cout + 127) / 128, 128, 0, s>>>(out, in, b, b2, w2, pin, Cin2, Cout);
    return cudaGetLastError();
}
cudaError_t launch_fill_rows(float* dst, const float* src, int C, int B, cudaStream_t s) {
    const int n = C * B;
    fill_rows_kernel<<<(n + 255) / 256, 256, 0, s>>>(dst, src, C, B);
    return cudaGetLastError();
}

cudaError_t launch_to_f32(const void* src, int dtype, float* dst, int64_t n, cudaStream_t s) {
    if (dtype == VD_BF16) to_f32_kernel<__nv_bfloat16><<<grid_for(n, 256), 256, 0, s>>>((const __nv_bfloat16*)src, dst, n);
    else to_f32_kernel<float><<<grid_for(n, 256), 256, 0, s>>>((const float*)src, dst, n);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// GroupNorm statistics without any caller-provided or allocated scratch memory.
//
// Some callers may not allocate device memory at the point where they need this operator: a
// render/game loop that must not stall on the allocator's implicit device synchronisation, a
// plug-in whose host application owns the whole memory pool, or code running where the CUDA
// allocator is simply off limits (inside a host callback, after a memory budget was frozen).
// For them the chunk partials of the reduction live in the fixed device array below instead of a
// buffer passed in.  The price is a size limit and shared state: every GPU that loads this
// library carries the array (148 KiB) until the process exits, and all calls on a device use the
// same array, so two calls whose kernels can overlap on the GPU (different streams, no ordering
// between them) race on it.  The chunk records need no clearing (every record read was written
// by the same call); the arrival counters behind them must start at zero and are cleared by an
// asynchronous memset at the start of every call.
namespace {
constexpr int kStaticGnMaxBatchTimesGroups = 64;     // e.g. 2 frames x 32 groups, or 8 x 8
constexpr int kStaticGnCounters = 64;                // arrival counters behind the records (batch <= 64 follows from the limit)
static __device__ __align__(256) float g_gn_static_partial[kStaticGnMaxBatchTimesGroups * kGnMaxChunks * 2 + kStaticGnCounters];   // 148 KiB of chunk records + 64 arrival counters

std::mutex g_static_mu;
constexpr int kMaxDevices = 64;
float* g_static_ptr[kMaxDevices] = {};

// In host code the array's name is only a handle of the symbol, not a device address; the address
// on the current device is looked up once per device and cached.
cudaError_t static_scratch_of_current_device(float** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_gn_static_partial);
        if (e != cudaSuccess) return e;
        g_static_ptr[dev] = (float*)p;
    }
    *out = g_static_ptr[dev];
    return cudaSuccess;
}
}  // namespace

}  // namespace vd

extern "C" VD_API vd_status vd_op_gn_stats_static(const void* x, int32_t dtype, int32_t batch, int32_t h, int32_t w,
                                                  int32_t c, int32_t groups, float eps, const float* gamma,
                                                  const float* beta, float* scale, float* shift, void* cuda_stream) {
    using namespace vd;
    if (!x || !gamma || !beta || !scale || !shift) { set_last_error("vd_op_gn_stats_static: NULL pointer"); return VD_ERR_INVALID_ARG; }
    if (dtype != VD_F32 && dtype != VD_BF16) { set_last_error("vd_op_gn_stats_static: bad dtype"); return VD_ERR_INVALID_ARG; }
    if (batch < 0 || h < 1 || w < 1 || c < 1 || groups < 1 || c % groups != 0 || (c / groups) % 4 != 0 || c > 1024) {
        set_last_error("vd_op_gn_stats_static: bad GroupNorm sizes (groups must hold a multiple of 4 channels)");
        return VD_ERR_INVALID_ARG;
    }
    if ((long long)h * w > 0x7fffffffLL || (long long)batch * h * w * c > (1LL << 40)) {
        set_last_error("vd_op_gn_stats_static: tensor too large (h*w must fit 31 bits, batch*h*w*c 40 bits)");
        return VD_ERR_INVALID_ARG;
    }
    if ((long long)batch * groups > kStaticGnMaxBatchTimesGroups) {
        set_last_error("vd_op_gn_stats_static: batch*groups exceeds 64, the capacity of the built-in scratch array; "
                       "use vd_op_gn_stats with a scratch buffer instead");
        return VD_ERR_UNSUPPORTED;
    }
    if (batch == 0) return VD_OK;
    float* partial = nullptr;
    cudaError_t e = static_scratch_of_current_device(&partial);
    if (e == cudaSuccess) {
        // the arrival counters live behind the records; they must be zero when the kernel starts
        unsigned int* counters = (unsigned int*)(partial + (size_t)kStaticGnMaxBatchTimesGroups * kGnMaxChunks * 2);
        e = cudaMemsetAsync(counters, 0, kStaticGnCounters * sizeof(unsigned int), (cudaStream_t)cuda_stream);
        GnArgs a{x, dtype, batch, h * w, c, groups, eps, gamma, beta, scale, shift, partial, counters, nullptr};
        if (e == cudaSuccess) e = launch_gn_stats(a, (cudaStream_t)cuda_stream);
    }
    if (e != cudaSuccess) {
        set_last_error((std::string("vd_op_gn_stats_static: ") + cudaGetErrorString(e)).c_str());
        return VD_ERR_CUDA;
    }
    return VD_OK;
}
