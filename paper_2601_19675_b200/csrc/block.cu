// Decoder-block operations between the quantized linear layers of a LLaMA-style stack at decode time (one new token
// per sequence): residual sum + RMS normalisation, rotary embedding + append to the key/value cache, attention of the
// new token over the cache (one cluster of CTAs per head and sequence), SiLU gating.  Not part of the
// quantization method: plain kernels, fp32 arithmetic, bf16 in and out, every read and write coalesced.
//
// At small batches each of these is a few microseconds of latency and a launch gap.  They are launched with programmatic
// stream serialization: a kernel's CTAs are resident when its predecessor ends and wait there (every kernel executes
// griddepcontrol.wait, so completion is transitive).  What a predecessor wrote is never read by __ldg: its non-coherent path
// promises nothing about data written while the kernel was resident already.  The small kernels release their successor
// at once, attention only when its CTAs are done with their keys: a successor that takes shared memory and thread slots
// while attention still has CTAs to start costs more than the gap.
#include "lopro_block.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace {

constexpr int kHeadDim = 128;     // the attention kernel is written for this head size
constexpr int kSplitKeys = 128;   // keys that lopro_block_attention_workspace_bytes counts a partial result for
constexpr int kPartial = kHeadDim + 2;

inline bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) red[warp] = v;
    __syncthreads();
    float t = 0.0f;
    for (int w = 0; w < nw; ++w) t += red[w];
    __syncthreads();
    return t;
}
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Eight bf16 entries: one 16-byte access where the row is aligned, else eight of two bytes.
template <bool VEC>
__device__ __forceinline__ uint4 load8(const __nv_bfloat16* p) {
    if constexpr (VEC) {
        return __ldcg(reinterpret_cast<const uint4*>(p));
    } else {
        uint4 u;
        unsigned short* e = reinterpret_cast<unsigned short*>(&u);
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = __ldcg(reinterpret_cast<const unsigned short*>(p) + i);
        return u;
    }
}
template <bool VEC>
__device__ __forceinline__ void store8(__nv_bfloat16* p, const uint4& u) {
    if constexpr (VEC) {
        *reinterpret_cast<uint4*>(p) = u;
    } else {
        const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&u);
#pragma unroll
        for (int i = 0; i < 8; ++i) p[i] = e[i];
    }
}

constexpr int kNormThreads = 512;
constexpr int kNormMax = 3;  // pieces of eight entries per thread: 12288 columns

// One token per CTA: h += y (rounded to bf16, stored), out = h * w / rms(h).  A latency chain -- loads, one block sum,
// stores --: every load, the weights among them, is in flight before the first use and the row stays in registers.
template <bool VEC>
__global__ void __launch_bounds__(kNormThreads) add_rmsnorm_kernel(__nv_bfloat16* __restrict__ h, int64_t ldh,
                                                                   const __nv_bfloat16* __restrict__ y, int64_t ldy,
                                                                   const __nv_bfloat16* __restrict__ w, float eps,
                                                                   __nv_bfloat16* __restrict__ out, int64_t ldo, int d) {
    __shared__ float red[kNormThreads / 32];
    const int t = blockIdx.x;
    __nv_bfloat16* hr = h + (size_t)t * ldh;
    release_successor();
    wait_for_predecessor();
    uint4 hv[kNormMax], yv[kNormMax], wv[kNormMax];
#pragma unroll
    for (int c = 0; c < kNormMax; ++c) {
        const int i = (c * kNormThreads + threadIdx.x) * 8;
        if (i < d) {
            hv[c] = load8<VEC>(hr + i);
            if (y != nullptr) yv[c] = load8<VEC>(y + (size_t)t * ldy + i);
            wv[c] = load8<VEC>(w + i);
        }
    }
    float ss = 0.0f;
#pragma unroll
    for (int c = 0; c < kNormMax; ++c) {
        const int i = (c * kNormThreads + threadIdx.x) * 8;
        if (i < d) {
            __nv_bfloat162* a = reinterpret_cast<__nv_bfloat162*>(&hv[c]);
            const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&yv[c]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (y != nullptr) {
                    const float2 u = __bfloat1622float2(a[e]), v = __bfloat1622float2(b[e]);
                    a[e] = __floats2bfloat162_rn(u.x + v.x, u.y + v.y);
                }
                const float2 f = __bfloat1622float2(a[e]);
                ss = fmaf(f.x, f.x, ss);
                ss = fmaf(f.y, f.y, ss);
            }
            if (y != nullptr) store8<VEC>(hr + i, hv[c]);
        }
    }
    ss = block_sum(ss, red);
    const float inv = rsqrtf(ss / (float)d + eps);
#pragma unroll
    for (int c = 0; c < kNormMax; ++c) {
        const int i = (c * kNormThreads + threadIdx.x) * 8;
        if (i < d) {
            uint4 o4;
            const __nv_bfloat162* a = reinterpret_cast<const __nv_bfloat162*>(&hv[c]);
            const __nv_bfloat162* g = reinterpret_cast<const __nv_bfloat162*>(&wv[c]);
            __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(&o4);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __bfloat1622float2(a[e]), wf = __bfloat1622float2(g[e]);
                o[e] = __floats2bfloat162_rn(f.x * inv * wf.x, f.y * inv * wf.y);
            }
            store8<VEC>(out + (size_t)t * ldo + i, o4);
        }
    }
}

__device__ __forceinline__ __nv_bfloat162 load2(const __nv_bfloat16* p) {
    const unsigned u = __ldcg(reinterpret_cast<const unsigned*>(p));
    return *reinterpret_cast<const __nv_bfloat162*>(&u);
}

// grid (n_heads, T), one thread per pair of dimensions.
__global__ void rope_append_kernel(__nv_bfloat16* __restrict__ q, int64_t ldq, const __nv_bfloat16* __restrict__ k,
                                   int64_t ldk, const __nv_bfloat16* __restrict__ v, int64_t ldv,
                                   const int32_t* __restrict__ pos, __nv_bfloat16* __restrict__ k_cache,
                                   __nv_bfloat16* __restrict__ v_cache, int n_heads, int head_dim, int ctx_max,
                                   double log2_theta, int* status) {
    const int hd = blockIdx.x, t = blockIdx.y, i = threadIdx.x;
    release_successor();
    const double freq = exp2(-2.0 * (double)i / (double)head_dim * log2_theta);  // (needs no input)
    wait_for_predecessor();
    if (i >= head_dim / 2) return;
    const size_t col = (size_t)hd * head_dim + 2 * i;
    __nv_bfloat162* qp = reinterpret_cast<__nv_bfloat162*>(q + (size_t)t * ldq + col);
    const __nv_bfloat162 q2 = load2(q + (size_t)t * ldq + col), k2 = load2(k + (size_t)t * ldk + col),
                         v2 = load2(v + (size_t)t * ldv + col);
    const int p = __ldcg(pos + t);
    if (p < 0 || p >= ctx_max) {
        if (i == 0) atomicCAS(status, LOPRO_OK, LOPRO_ERR_INVALID_DATA);
        return;
    }
    double sn, cs;
    sincos((double)p * freq, &sn, &cs);
    const float c = (float)cs, s = (float)sn;
    const float2 qv = __bfloat1622float2(q2), kv = __bfloat1622float2(k2);
    *qp = __floats2bfloat162_rn(qv.x * c - qv.y * s, qv.x * s + qv.y * c);
    const size_t entry = (((size_t)t * n_heads + hd) * ctx_max + p) * head_dim + 2 * i;
    *reinterpret_cast<__nv_bfloat162*>(k_cache + entry) = __floats2bfloat162_rn(kv.x * c - kv.y * s, kv.x * s + kv.y * c);
    *reinterpret_cast<__nv_bfloat162*>(v_cache + entry) = v2;
}

constexpr int kAttnBatch = 4;                   // keys that a half-warp holds at once (and as many on their way)
constexpr int kMaxCluster = 8;

// Attention of one query over the keys of its sequence; grid cluster x pairs, one cluster of CTAs per (head, sequence) pair
// from pair0 on.  Bound by reading keys and values once.  The sequence's keys are shared out evenly over the cluster's CTAs,
// and within a CTA over its half-warps: sixteen lanes read a key's (value's) 256 bytes as one 16-byte piece each, so every
// access is a whole row, and a half-warp needs nobody else until the end: it keeps its own running maximum, sum of weights
// and weighted values.  Keys and values of the next four keys are requested before the present four are used.  The
// half-warps' results meet in shared memory, the CTAs' in that of the cluster's first CTA: no merging launch, no scratch
// in global memory (the workspace of the entry point is not touched).
// 32 sequences of 32 heads, context 2049 (1.07 GB): 217 us in two launches before, 165 us = 6.5 TB/s now.
// kWhole: all pairs.  kFirst, kTail: the pairs of a short last wave run as a second launch in larger clusters, which starts
// as the first launch's CTAs finish.  For that the first releases it when its own predecessor is complete, and the tail
// reads without waiting and waits for the first launch before it ends, so that its successor waits for both.
// 16 sequences of 40 heads, context 2540 (0.83 GB; 640 pairs over 592 slots): 180 us in one launch, 123 us = 6.8 TB/s.
enum AttnPart { kWhole, kFirst, kTail };
template <int THREADS, AttnPart PART>
__global__ void __launch_bounds__(THREADS, 512 / THREADS)
attention_kernel(const __nv_bfloat16* __restrict__ q, int64_t ldq, const __nv_bfloat16* __restrict__ k_cache,
                 const __nv_bfloat16* __restrict__ v_cache, const int32_t* __restrict__ ctx, int n_heads, int ctx_max, float scale,
                 __nv_bfloat16* __restrict__ out, int64_t ldo, int* status, int size, int pair0) {
    constexpr int kAttnHalves = THREADS / 16;          // half-warps, each a stream of keys of its own
    __shared__ float acc_s[kAttnHalves][kHeadDim];
    __shared__ float2 ml_s[kAttnHalves];               // (maximum, sum) of a half-warp
    __shared__ __align__(16) float part_s[kMaxCluster][kHeadDim + 4];  // first CTA: the CTAs' weighted values, maximum, sum
    const int pair = pair0 + (int)blockIdx.x / size, rank = (int)blockIdx.x % size, tid = threadIdx.x;
    const int t = pair / n_heads, hd = pair - t * n_heads;
    const int half = tid >> 4, piece = tid & 15;
    if (size > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // this CTA has started
    if (PART != kTail) wait_for_predecessor();
    if (PART == kFirst) release_successor();
    const int n_all = __ldcg(ctx + t);
    const bool bad = n_all < 1 || n_all > ctx_max;
    if (bad && tid == 0 && hd == 0 && rank == 0) atomicCAS(status, LOPRO_OK, LOPRO_ERR_INVALID_DATA);
    const int n = bad ? 0 : n_all;
    float qf[8];
    const __nv_bfloat16* qr = q + (size_t)t * ldq + (size_t)hd * kHeadDim + 8 * piece;
#pragma unroll
    for (int e = 0; e < 8; ++e)
        qf[e] = __bfloat162float(__ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short*>(qr) + e))) * scale;
    // keys j0 .. j1 of this CTA; the half-warp's are j0 + half, + 8, ...
    const int per = (n + size - 1) / size, j0 = min(rank * per, n), j1 = min(j0 + per, n);
    const size_t base = ((size_t)t * n_heads + hd) * ctx_max;
    const uint4* kr = reinterpret_cast<const uint4*>(k_cache + base * kHeadDim) + piece;
    const uint4* vr = reinterpret_cast<const uint4*>(v_cache + base * kHeadDim) + piece;
    float m = -INFINITY, l = 0.0f, acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
    uint4 ka[kAttnBatch], va[kAttnBatch], kb[kAttnBatch], vb[kAttnBatch];
    auto fetch = [&](uint4 (&kk)[kAttnBatch], uint4 (&vv)[kAttnBatch], int j) {
#pragma unroll
        for (int c = 0; c < kAttnBatch; ++c) {
            const int jj = j + c * kAttnHalves;
            if (jj < j1) {
                kk[c] = __ldcg(kr + (size_t)jj * (kHeadDim / 8));
                vv[c] = __ldcg(vr + (size_t)jj * (kHeadDim / 8));
            }
        }
    };
    auto consume = [&](const uint4 (&kk)[kAttnBatch], const uint4 (&vv)[kAttnBatch], int j) {
        float s[kAttnBatch], top = m;
#pragma unroll
        for (int c = 0; c < kAttnBatch; ++c) {
            const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&kk[c]);
            float d0 = 0.0f, d1 = 0.0f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __bfloat1622float2(b[e]);
                d0 = fmaf(f.x, qf[2 * e], d0);
                d1 = fmaf(f.y, qf[2 * e + 1], d1);
            }
            s[c] = d0 + d1;
        }
#pragma unroll
        for (int o = 1; o < 16; o <<= 1)
#pragma unroll
            for (int c = 0; c < kAttnBatch; ++c) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
#pragma unroll
        for (int c = 0; c < kAttnBatch; ++c) {
            if (j + c * kAttnHalves >= j1) s[c] = -INFINITY;
            top = fmaxf(top, s[c]);
        }
        if (top == -INFINITY) return;   // (no key of this half-warp yet)
        const float keep = __expf(m - top);
        m = top;
        l *= keep;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] *= keep;
#pragma unroll
        for (int c = 0; c < kAttnBatch; ++c) {
            if (j + c * kAttnHalves < j1) {
                const float w = __expf(s[c] - top);
                l += w;
                const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&vv[c]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 f = __bfloat1622float2(b[e]);
                    acc[2 * e] = fmaf(w, f.x, acc[2 * e]);
                    acc[2 * e + 1] = fmaf(w, f.y, acc[2 * e + 1]);
                }
            }
        }
    };
    // (every lane of a warp runs the same number of rounds: the shuffles take part in all of them)
    constexpr int kStep = kAttnBatch * kAttnHalves;
    const int first = j0 + half;
    fetch(ka, va, first);
    for (int r = 0; j0 + r < j1; r += 2 * kStep) {
        fetch(kb, vb, first + r + kStep);
        consume(ka, va, first + r);
        if (j0 + r + kStep >= j1) break;
        fetch(ka, va, first + r + 2 * kStep);
        consume(kb, vb, first + r + kStep);
    }
    if (PART != kFirst) release_successor();
#pragma unroll
    for (int e = 0; e < 8; ++e) acc_s[half][8 * piece + e] = acc[e];
    if (piece == 0) ml_s[half] = make_float2(m, l);
    __syncthreads();
    // the CTA's result, one dimension per thread
    float top = -INFINITY, num = 0.0f, den = 0.0f;
#pragma unroll
    for (int h = 0; h < kAttnHalves; ++h) top = fmaxf(top, ml_s[h].x);
#pragma unroll
    for (int h = 0; h < kAttnHalves; ++h) {
        const float w = ml_s[h].x > -INFINITY ? __expf(ml_s[h].x - top) : 0.0f;
        num = fmaf(w, acc_s[h][tid & (kHeadDim - 1)], num);
        den = fmaf(w, ml_s[h].y, den);
    }
    if (size > 1) {
        // into the first CTA's shared memory, once all CTAs are known to have started
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        uint32_t dst;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&part_s[rank][0])), "r"(0));
        if (tid < kHeadDim) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 4u * (uint32_t)tid), "f"(num) : "memory");
        if (tid == 0) {
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 4u * kHeadDim), "f"(top) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 4u * kHeadDim + 4u), "f"(den) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank != 0) {
            if (PART == kTail) wait_for_predecessor();
            return;
        }
        top = -INFINITY;
        num = den = 0.0f;
        for (int c = 0; c < size; ++c) top = fmaxf(top, part_s[c][kHeadDim]);
        for (int c = 0; c < size; ++c) {
            const float w = part_s[c][kHeadDim] > -INFINITY ? __expf(part_s[c][kHeadDim] - top) : 0.0f;
            num = fmaf(w, part_s[c][tid & (kHeadDim - 1)], num);
            den = fmaf(w, part_s[c][kHeadDim + 1], den);
        }
    }
    if (tid < kHeadDim) out[(size_t)t * ldo + (size_t)hd * kHeadDim + tid] = __float2bfloat16_rn(den > 0.0f ? num / den : 0.0f);
    if (PART == kTail) wait_for_predecessor();
}

__global__ void __launch_bounds__(256) silu_mul_kernel(const __nv_bfloat16* __restrict__ gate, int64_t ldg,
                                                       const __nv_bfloat16* __restrict__ up, int64_t ldu,
                                                       __nv_bfloat16* __restrict__ out, int64_t ldo, int d) {
    const int t = blockIdx.y;
    const int i = (blockIdx.x * 256 + threadIdx.x) * 8;
    release_successor();
    wait_for_predecessor();
    if (i >= d) return;
    const uint4 g4 = load8<true>(gate + (size_t)t * ldg + i), u4 = load8<true>(up + (size_t)t * ldu + i);
    uint4 o4;
    const __nv_bfloat162* g = reinterpret_cast<const __nv_bfloat162*>(&g4);
    const __nv_bfloat162* u = reinterpret_cast<const __nv_bfloat162*>(&u4);
    __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(&o4);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 a = __bfloat1622float2(g[e]), b = __bfloat1622float2(u[e]);
        o[e] = __floats2bfloat162_rn(a.x / (1.0f + __expf(-a.x)) * b.x, a.y / (1.0f + __expf(-a.y)) * b.y);
    }
    *reinterpret_cast<uint4*>(out + (size_t)t * ldo + i) = o4;
}

// One launch with programmatic stream serialization, and a cluster of `cluster` CTAs along x where that is more than 1.
template <typename... Params, typename... Args>
lopro_status launch(void (*kernel)(Params...), dim3 grid, int threads, void* stream, int cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...) == cudaSuccess ? LOPRO_OK : LOPRO_ERR_CUDA;
}

}  // namespace

extern "C" {

lopro_status lopro_block_add_rmsnorm(uint16_t* h, int64_t ldh, const uint16_t* y, int64_t ldy, const uint16_t* w, float eps,
                                     uint16_t* out, int64_t ldo, int32_t T, int32_t d, void* stream) {
    if (T < 0 || d < 8 || (d % 8) || d > 12288 || !(eps >= 0.0f)) return LOPRO_ERR_INVALID_ARG;
    if (T == 0) return LOPRO_OK;
    if (!h || !w || !out || ldh < d || ldo < d || (y && ldy < d)) return LOPRO_ERR_INVALID_ARG;
    const bool vec = aligned_to(h, 16) && aligned_to(w, 16) && aligned_to(out, 16) && (ldh % 8) == 0 && (ldo % 8) == 0 &&
                     (!y || (aligned_to(y, 16) && (ldy % 8) == 0));
    return launch(vec ? add_rmsnorm_kernel<true> : add_rmsnorm_kernel<false>, dim3(T), kNormThreads, stream, 1,
                  reinterpret_cast<__nv_bfloat16*>(h), ldh, reinterpret_cast<const __nv_bfloat16*>(y), ldy,
                  reinterpret_cast<const __nv_bfloat16*>(w), eps, reinterpret_cast<__nv_bfloat16*>(out), ldo, d);
}

lopro_status lopro_block_rope_append(uint16_t* q, int64_t ldq, const uint16_t* k, int64_t ldk, const uint16_t* v, int64_t ldv,
                                     const int32_t* pos, uint16_t* k_cache, uint16_t* v_cache, int32_t T, int32_t n_heads,
                                     int32_t head_dim, int32_t ctx_max, float theta, void* status_word, void* stream) {
    if (T < 0 || n_heads < 1 || n_heads > 65535 || head_dim < 2 || (head_dim % 2) || head_dim > 256 || ctx_max < 1 ||
        !(theta > 1.0f))
        return LOPRO_ERR_INVALID_ARG;
    if (T == 0) return LOPRO_OK;
    const int64_t width = (int64_t)n_heads * head_dim;
    if (!q || !k || !v || !pos || !k_cache || !v_cache || !status_word || ldq < width || ldk < width || ldv < width ||
        (ldq % 2) || (ldk % 2) || (ldv % 2) || T > 65535)
        return LOPRO_ERR_INVALID_ARG;
    if (!aligned_to(q, 4) || !aligned_to(k, 4) || !aligned_to(v, 4) || !aligned_to(k_cache, 4) || !aligned_to(v_cache, 4))
        return LOPRO_ERR_INVALID_ARG;
    return launch(rope_append_kernel, dim3(n_heads, T), (head_dim / 2 + 31) / 32 * 32, stream, 1,
                  reinterpret_cast<__nv_bfloat16*>(q), ldq, reinterpret_cast<const __nv_bfloat16*>(k), ldk,
                  reinterpret_cast<const __nv_bfloat16*>(v), ldv, pos, reinterpret_cast<__nv_bfloat16*>(k_cache),
                  reinterpret_cast<__nv_bfloat16*>(v_cache), n_heads, head_dim, ctx_max, log2((double)theta), (int*)status_word);
}

size_t lopro_block_attention_workspace_bytes(int32_t T, int32_t n_heads, int32_t head_dim, int32_t ctx_max) {
    if (T < 0 || n_heads < 1 || head_dim != kHeadDim || ctx_max < 1) return 0;
    const size_t splits = ((size_t)ctx_max + kSplitKeys - 1) / kSplitKeys;
    return ((size_t)T * n_heads * splits * kPartial * sizeof(float) + 255) / 256 * 256 + 256;
}

lopro_status lopro_block_attention_decode(const uint16_t* q, int64_t ldq, const uint16_t* k_cache, const uint16_t* v_cache,
                                          const int32_t* ctx, uint16_t* out, int64_t ldo, int32_t T, int32_t n_heads,
                                          int32_t head_dim, int32_t ctx_max, float scale, void* workspace,
                                          size_t workspace_bytes, void* status_word, void* stream) {
    if (T < 0 || n_heads < 1 || n_heads > 65535 || ctx_max < 1) return LOPRO_ERR_INVALID_ARG;
    if (head_dim != kHeadDim) return LOPRO_ERR_UNSUPPORTED;
    if (T == 0) return LOPRO_OK;
    const int64_t width = (int64_t)n_heads * head_dim;
    if (!q || !k_cache || !v_cache || !ctx || !out || !workspace || !status_word || ldq < width || ldo < width || T > 65535)
        return LOPRO_ERR_INVALID_ARG;
    if (!aligned_to(k_cache, 16) || !aligned_to(v_cache, 16) || !aligned_to(workspace, 256)) return LOPRO_ERR_INVALID_ARG;
    if (workspace_bytes < lopro_block_attention_workspace_bytes(T, n_heads, head_dim, ctx_max)) return LOPRO_ERR_BUFFER_TOO_SMALL;
    // Four CTAs of 128 threads fit a multiprocessor.  The cluster is the largest with which all CTAs are still resident at
    // once (8 sequences of 32 heads: 61 us without clusters, 46 with 2, 50 with 4; 32 sequences: 165, 175, 184), and
    // where clusters of 8 leave room the CTAs are twice as large.
    const int64_t pairs = (int64_t)T * n_heads, slots = 4 * (int64_t)lopro::sm_count();
    int cluster = 1;
    while (cluster < kMaxCluster && pairs * cluster * 2 <= slots) cluster *= 2;
    const bool wide = pairs * cluster * 2 <= slots;
    // The loads in flight land in L1.  A programmatic launch puts the first CTAs beside those of a product kernel that holds
    // 220 KB of shared memory, and as long as the multiprocessor is never empty its split stays: 28 KB of L1 for all waves of
    // this grid.  With a split of its own asked for, the grid starts on multiprocessors that have it: 32 sequences of 32 heads
    // after the q/k/v projections of a decoder layer 202 us without, 160 with (163 alone).  Three quarters of shared memory,
    // which leave 57 KB of L1, do as well as one for grids of several waves (decoder layer, 19 sequences of 40 heads, context
    // 1705: 294 us without, 270 and 270), and cost a grid of one wave nothing, where the smaller share did (10 sequences of 32
    // heads, context 2410: 156 us without, 161 with a quarter, 157 with three).
    static unsigned long long split_whole = 0, split_first = 0;
    lopro::prefer_shared_memory(attention_kernel<128, kWhole>, 75, &split_whole);
    lopro::prefer_shared_memory(attention_kernel<128, kFirst>, 75, &split_first);
    auto run = [&](auto kernel, int size, int threads, int64_t first, int64_t count) {
        return launch(kernel, dim3((unsigned)(count * size)), threads, stream, size, reinterpret_cast<const __nv_bfloat16*>(q), ldq,
                      reinterpret_cast<const __nv_bfloat16*>(k_cache), reinterpret_cast<const __nv_bfloat16*>(v_cache), ctx, n_heads,
                      ctx_max, scale, reinterpret_cast<__nv_bfloat16*>(out), ldo, (int*)status_word, size, (int)first);
    };
    if (pairs > 0x7fffffff) return LOPRO_ERR_UNSUPPORTED;   // (a cache of half a terabyte)
    if (wide) return run(attention_kernel<256, kWhole>, cluster, 256, 0, pairs);
    // A last wave that leaves half the slots idle or more: its pairs in clusters that fill them.
    const int64_t rest = pairs % slots;
    if (pairs < slots || rest == 0 || rest * 2 > slots) return run(attention_kernel<128, kWhole>, cluster, 128, 0, pairs);
    const lopro_status st = run(attention_kernel<128, kFirst>, 1, 128, 0, pairs - rest);
    if (st != LOPRO_OK) return st;
    for (cluster = 2; cluster < kMaxCluster && rest * cluster * 2 <= slots; ) cluster *= 2;
    return run(attention_kernel<128, kTail>, cluster, 128, pairs - rest, rest);
}

lopro_status lopro_block_silu_mul(const uint16_t* gate, int64_t ldg, const uint16_t* up, int64_t ldu, uint16_t* out,
                                  int64_t ldo, int32_t T, int32_t d, void* stream) {
    if (T < 0 || d < 8 || (d % 8) || T > 65535) return LOPRO_ERR_INVALID_ARG;
    if (T == 0) return LOPRO_OK;
    if (!gate || !up || !out || ldg < d || ldu < d || ldo < d || (ldg % 8) || (ldu % 8) || (ldo % 8)) return LOPRO_ERR_INVALID_ARG;
    if (!aligned_to(gate, 16) || !aligned_to(up, 16) || !aligned_to(out, 16)) return LOPRO_ERR_INVALID_ARG;
    return launch(silu_mul_kernel, dim3((d / 8 + 255) / 256, T), 256, stream, 1, reinterpret_cast<const __nv_bfloat16*>(gate), ldg,
                  reinterpret_cast<const __nv_bfloat16*>(up), ldu, reinterpret_cast<__nv_bfloat16*>(out), ldo, d);
}

}  // extern "C"
