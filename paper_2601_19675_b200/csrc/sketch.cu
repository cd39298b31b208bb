// Rank-1 randomized sketch with deflation (Sec. 3.3, Eq. 10-12; inner loop of Algorithm 1) as ONE persistent kernel.
//
// What bounds it: reading the fp32 matrix.  Per rank the method forms y = (W W^T)^it W v and p = W^T y, 2 it + 2
// matrix-vector products, then W <- W - sigma u v^T.  Two things keep W from being touched more often than it must:
//  * A product pair p = W^T (W v) needs a row of W once: the row's dot product with v gives y_i, and y_i times the same
//    row goes into p while the row is still in registers: it + 1 passes per rank instead of 2 it + 2.
//  * W is never rewritten.  With W_j = W diag(s) - sum_{l<j} sigma_l u_l v_l^T,
//        W_j v = W (s v) - sum_l sigma_l (v_l v) u_l,     W_j^T y = s (W^T y) - sum_l sigma_l (u_l y) v_l,
//    a few scalars per rank instead of a read and a write of the matrix.
//
// Layout: one CTA of 512 threads per SM owns a contiguous run of rows for the whole computation.  A stage of R rows is
// spread over TR threads, V float4 columns each (short rows: G = 512 / TR groups with stages of their own).  A row costs a
// reduction over its threads between its two products; the loop is pipelined so that a stage's second product runs while
// the next stage's first one is reduced (both held in registers), one barrier per stage.  Stages arrive by bulk copies in a
// ring of shared memory that runs ahead across the passes, so the two grid barriers of a pass (partial sums written; sums
// formed) pass with copies in flight.  Where a CTA's rows fit the ring they stay there and only the first pass reads memory.
// Successive passes walk the rows in opposite directions: what the last pass read last is still in L2.
//
// Measured (rank 16, 8 iterations, whole layer): 11008 x 4096 11.8 -> 4.8 ms, 7 us of each 31 us pass in the two barriers and
// the sums between them; while the rows stream 7.5 TB/s, of which HBM delivers about 60 % and L2, thanks to the turned
// direction, the rest (DRAM 43 % busy over the whole kernel); 4096 x 4096 3.9 -> 2.0 ms.
//
// All sums have a fixed order (threads, rows of a CTA, CTAs): the result depends on the number of CTAs, never on timing.
// Every wait is bounded.  One that runs out raises the abort flag before its CTA arrives at the next grid barrier.  The flag
// is a bit of the word that counts the arrivals, so no CTA gets past that barrier without it (a word of its own, read behind
// every barrier, cost 0.25 us each: 4096 x 512 at rank 8 327 -> 348 us).  All leave there, store LOPRO_ERR_TIMEOUT and let w be.
#include "common.cuh"
#include "ptx.cuh"
#include "sketch.cuh"

namespace lopro {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kRingBytes = 196 * 1024;
constexpr int kMaxCtas = 192;                  // multiprocessors the sums over CTAs are written for
constexpr int kMaxSlots = 64;                  // ring slots of all groups together
constexpr int kMaxRank = 128;                  // one thread of a row per rank before
constexpr int kMaxOwn = 32;                    // float4 columns of p a CTA sums
constexpr uint32_t kGridSpin = 1u << 24;       // polls of a grid barrier before it gives up
constexpr unsigned kAbort = 1u << 31;          // in the count of arrivals (2 (it + 1) r barriers of at most 192 CTAs: 22 bits)

struct SketchParams {
    const float* w;         // [m][n]
    const float* sketches;  // [r][n]
    const float* s;         // column scale, or null
    float* s_eff;           // [n] the scale as applied (null: none wanted)
    __half* s16;            // [n] the scale as stored (null: not rounded)
    float *U, *sigma, *V;
    float* y;               // [m]
    float* p;               // [n]
    float* partial;         // [gridDim][n] sums of y_i w_i
    float* ext_rows;        // [1 + r][gridDim]: |y|^2, u_l y   (sums over rows)
    float* ext_cols;        // [1 + r][gridDim]: |p|^2, v_l p   (sums over columns)
    unsigned* sync;         // arrivals and the abort flag; zero at launch
    int* status;
    int m, n, r, it, cast;
    int slots;              // ring slots per group
    int resident;           // every group's stages fit its slots
};

__device__ __forceinline__ float inv_norm(float sumsq) {
    const float nrm = sqrtf(sumsq);
    return (nrm > 0.0f && isfinite(nrm)) ? 1.0f / nrm : 0.0f;
}
__device__ __forceinline__ void group_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void axpy(float4& acc, float a, const float4& v) {
    acc.x = fmaf(a, v.x, acc.x);
    acc.y = fmaf(a, v.y, acc.y);
    acc.z = fmaf(a, v.z, acc.z);
    acc.w = fmaf(a, v.w, acc.w);
}
// element-wise partial dot products: four chains
__device__ __forceinline__ void dot4(float4& acc, const float4& a, const float4& b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.y = fmaf(a.y, b.y, acc.y);
    acc.z = fmaf(a.z, b.z, acc.z);
    acc.w = fmaf(a.w, b.w, acc.w);
}
// Four columns as two pairs: one fused multiply-add instruction per pair (each lane of it rounds as a plain one).
struct Quad {
    unsigned long long lo, hi;
};
__device__ __forceinline__ unsigned long long pair(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float pair_sum(unsigned long long v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a + b;
}
__device__ __forceinline__ unsigned long long pair_fma(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ Quad quad(const float4& v) { return Quad{pair(v.x, v.y), pair(v.z, v.w)}; }
__device__ __forceinline__ Quad load_quad(const Quad* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return Quad{v.x, v.y};
}
__device__ __forceinline__ float sum4(const float4& a) { return (a.x + a.y) + (a.z + a.w); }
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// sum over the CTAs of one row of an ext array, by a warp
__device__ __forceinline__ float cta_sum(const float* row, int ctas, int lane) {
    float t[kMaxCtas / 32], a = 0.0f;
#pragma unroll
    for (int e = 0; e < kMaxCtas / 32; ++e) t[e] = lane + 32 * e < ctas ? __ldcg(row + lane + 32 * e) : 0.0f;
#pragma unroll
    for (int e = 0; e < kMaxCtas / 32; ++e) a += t[e];
    return warp_sum(a);
}
__device__ __forceinline__ float4 cast4(const float4& v, float f, int cast) {
    float4 o = make_float4(f * v.x, f * v.y, f * v.z, f * v.w);
    if (cast) o = make_float4(round_e4m3(o.x), round_e4m3(o.y), round_e4m3(o.z), round_e4m3(o.w));
    return o;
}
// the scale of four columns, as applied
__device__ __forceinline__ float4 scale_of(const SketchParams& p, int col) {
    float4 t = make_float4(1.f, 1.f, 1.f, 1.f);
    if (p.s != nullptr) t = make_float4(__ldg(p.s + 4 * col), __ldg(p.s + 4 * col + 1), __ldg(p.s + 4 * col + 2), __ldg(p.s + 4 * col + 3));
    if (p.s16 != nullptr)
        t = make_float4(__half2float(__float2half_rn(t.x)), __half2float(__float2half_rn(t.y)), __half2float(__float2half_rn(t.z)),
                        __half2float(__float2half_rn(t.w)));
    return t;
}

// TR threads per row, V float4 columns per thread (4 TR V >= n), R rows per stage.
template <int TR, int V, int R>
__global__ void __launch_bounds__(kThreads, 1) sketch_kernel(const SketchParams p) {
    constexpr int G = kThreads / TR, W = TR / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[kMaxSlots];
    constexpr int P = 32 / R;                          // P lanes work on a row's sum
    constexpr int NV = W * R >= 32 ? W * R / 32 : 1;   // warps' sums that a lane adds
    __shared__ __align__(16) float red[G][2][R * W];   // row dot products by warp, two stages
    __shared__ float sig[kMaxRank];                   // sigma_l
    __shared__ float coef[kMaxRank + 1];              // sigma_l (v_l v), then sigma_l (u_l y)
    __shared__ float s_vv, s_yy;                      // |v|^2 (|p|^2 at the end of a rank), |y|^2
    __shared__ float part[G][kMaxRank + 1];           // per group: |y|^2, u_l y
    __shared__ float dots[kMaxRank + 1][kWarps];      // v_l v by warp for the sketch vector
    __shared__ __align__(16) float4 gsum[G > 1 ? (G - 1) * TR * V : 1];   // the groups' sums of p
    __shared__ __align__(16) float4 colred[64][9];
    __shared__ __align__(16) float4 own[kMaxOwn];     // this CTA's columns of p
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = tid / TR, tg = tid % TR, warp = tg >> 5;
    const int n = p.n, n4 = n >> 2, ctas = (int)gridDim.x, cta = (int)blockIdx.x;
    // the CTA's rows, the group's stages among them, the CTA's columns of p
    const int base = p.m / ctas, extra = p.m - base * ctas;
    const int row0 = cta * base + min(cta, extra), rows = base + (cta < extra ? 1 : 0);
    const int stages_all = (rows + R - 1) / R;
    const int SG = (stages_all - g + G - 1) / G;       // stages g, g + G, ... of the CTA
    const int per = (n4 + ctas - 1) / ctas, c0 = min(cta * per, n4), c1 = min(c0 + per, n4);
    const uint32_t stage_bytes = (uint32_t)(R * n * 4);
    unsigned char* ring = smem + (size_t)g * p.slots * stage_bytes;
    const uint32_t bar0 = smem_u32(bars) + 8u * (uint32_t)(g * p.slots);
    if (tid == 0) {
        for (int i = 0; i < G * p.slots; ++i) mbar_init(smem_u32(bars) + 8u * (uint32_t)i, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    const int n_pass = p.r * (p.it + 1);
    const int n_loads = p.resident ? SG : n_pass * SG;
    // the next copy of the group (its thread 0 counts along, with additions only: the group waits for it); the
    // direction turns with every pass
    int ahead_left = SG, ahead_st = g, ahead_step = G, ahead_slot = 0;
    auto issue = [&]() {
        const uint32_t bytes = (uint32_t)min(R, rows - ahead_st * R) * (uint32_t)(n * 4);
        const uint32_t bar = bar0 + 8u * (uint32_t)ahead_slot;
        mbar_expect_tx(bar, bytes);
        bulk_g2s(smem_u32(ring) + (uint32_t)ahead_slot * stage_bytes, p.w + (size_t)(row0 + ahead_st * R) * n, bytes, bar);
        ahead_st += ahead_step;
        if (--ahead_left == 0) {
            ahead_left = SG;
            ahead_st -= ahead_step;
            ahead_step = -ahead_step;
        }
        if (++ahead_slot == p.slots) ahead_slot = 0;
    };
    if (tg == 0)
        for (int i = 0; i < min(p.slots, n_loads); ++i) issue();
    if (cta == 0 && p.s_eff != nullptr)
        for (int c = tid; c < n4; c += kThreads) {
            const float4 t = scale_of(p, c);
            reinterpret_cast<float4*>(p.s_eff)[c] = t;
            if (p.s16 != nullptr) {
                p.s16[4 * c] = __float2half_rn(t.x);
                p.s16[4 * c + 1] = __float2half_rn(t.y);
                p.s16[4 * c + 2] = __float2half_rn(t.z);
                p.s16[4 * c + 3] = __float2half_rn(t.w);
            }
        }

    bool dead_wait = false;    // this thread's wait for a stage ran out: it waits for no other
    unsigned generation = 0;
    auto grid_sync = [&]() {  // false: some CTA gave up, all leave
        __syncthreads();
        ++generation;
        if (tid == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.sync) : "memory");
            const unsigned target = generation * (unsigned)ctas;
            unsigned seen;
            for (uint32_t i = 0; (seen = load_acquire(p.sync)) < target; ++i) {   // (the flag ends the wait too)
                if (i > kGridSpin) {
                    seen = kAbort | atomicOr(p.sync, kAbort);
                    break;
                }
            }
            if (seen & kAbort) s_abort = 1;
        }
        __syncthreads();
        return s_abort == 0;
    };

    // this thread's columns; those past the end of the row repeat its last four and meet a zero of v
    int cidx[V];
#pragma unroll
    for (int c = 0; c < V; ++c) cidx[c] = min(c * TR + tg, n4 - 1);
    int q = 0, slot = 0;  // stages consumed, ring slot of the next one
    uint32_t parity = 0;
    bool back = false;
    float ip = 0.0f;      // 1 / |p| of the rank before
    bool rank_dead = false;  // the rank before is a zero triple: its p may hold NaN or infinities, which no factor 0 removes
    int pass = 0;
    for (int j = 0; j < p.r; ++j) {
        for (int k = 0; k <= p.it; ++k, ++pass) {
            // ---- the vector of the pass, its norm and its products with the v_l ----
            float4 v[V];
            const float4* vsrc = reinterpret_cast<const float4*>(k == 0 ? p.sketches + (size_t)j * n : p.p);
#pragma unroll
            for (int c = 0; c < V; ++c) v[c] = c * TR + tg < n4 ? __ldcg(vsrc + cidx[c]) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (k > 0) {
                for (int l = wid; l <= j; l += kWarps) {
                    const float t = cta_sum(p.ext_cols + (size_t)l * ctas, ctas, lane);
                    if (lane == 0) {
                        if (l == 0) s_vv = t;
                        else coef[l - 1] = sig[l - 1] * t;
                    }
                }
            } else {
                // the sketch vector: every group takes some of the v_l (the last one is not stored everywhere yet: it is
                // p / |p| of the rank before)
                for (int l = g; l <= j; l += G) {   // l = 0: |v|^2; l > 0: v_{l-1} v
                    float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < V; ++c) {
                        float4 x;
                        if (l == 0) x = v[c];
                        else if (l == j) x = rank_dead ? make_float4(0.f, 0.f, 0.f, 0.f)
                                                       : cast4(__ldcg(reinterpret_cast<const float4*>(p.p) + cidx[c]), ip, p.cast);
                        else x = __ldcg(reinterpret_cast<const float4*>(p.V + (size_t)(l - 1) * n) + cidx[c]);
                        dot4(d, x, v[c]);
                    }
                    const float t = warp_sum(sum4(d));
                    if (lane == 0) dots[l][warp] = t;
                }
                __syncthreads();
                if (tid <= j) {
                    float t = 0.0f;
#pragma unroll
                    for (int w = 0; w < W; ++w) t += dots[tid][w];
                    if (tid == 0) s_vv = t;
                    else coef[tid - 1] = sig[tid - 1] * t;
                }
            }
            if (p.s != nullptr || p.s16 != nullptr) {
#pragma unroll
                for (int c = 0; c < V; ++c) {
                    const float4 t = scale_of(p, cidx[c]);
                    v[c] = make_float4(v[c].x * t.x, v[c].y * t.y, v[c].z * t.z, v[c].w * t.w);
                }
            }
            Quad vq[V], pacc[V];
#pragma unroll
            for (int c = 0; c < V; ++c) {
                vq[c] = quad(v[c]);
                pacc[c] = Quad{0ull, 0ull};
            }
            __syncthreads();
            const float inv_v = inv_norm(s_vv);
            const bool has_rank = warp * 32 < j;               // rank l = tg rides in this thread's part of the dot products
            const float my_coef = tg < j ? -coef[tg] : 0.0f;
            float sqsum = 0.0f, uy = 0.0f;

            // ---- the rows ----
            const int st0 = back ? (SG - 1) * G + g : g, st_step = back ? -G : G;
            // stage i: its rows into registers, their dot products with v, the warp's part of the sums to shared memory
            auto first_half = [&](int i, Quad (&w)[R][V], float (&u)[R]) {
                const int st = st0 + i * st_step, cnt = min(R, rows - st * R), r0 = row0 + st * R;
                if (has_rank)
#pragma unroll
                    for (int r = 0; r < R; ++r) u[r] = tg < j && r < cnt ? p.U[(size_t)(r0 + r) * p.r + tg] : 0.0f;
                if (p.resident) slot = st / G;
                if (!dead_wait && !mbar_wait(bar0 + 8u * (uint32_t)slot, parity)) {
                    dead_wait = true;
                    atomicOr(p.sync, kAbort);
                }
                const Quad* sm = reinterpret_cast<const Quad*>(ring + (size_t)slot * stage_bytes);
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int c = 0; c < V; ++c) w[r][c] = load_quad(sm + (r < cnt ? r : 0) * n4 + cidx[c]);
            };
            auto first_sums = [&](int i, const Quad (&w)[R][V], const float (&u)[R]) {
                float d[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    Quad a = {0ull, 0ull};
#pragma unroll
                    for (int c = 0; c < V; ++c) {
                        a.lo = pair_fma(w[r][c].lo, vq[c].lo, a.lo);
                        a.hi = pair_fma(w[r][c].hi, vq[c].hi, a.hi);
                    }
                    d[r] = pair_sum(a.lo) + pair_sum(a.hi);
                    if (has_rank) d[r] = fmaf(my_coef, u[r], d[r]);
                }
                // sums over the lanes, halving the rows a lane holds where there are several: lane / P ends with its row
#pragma unroll
                for (int h = R / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
                    const bool upper = (lane & o) != 0;
#pragma unroll
                    for (int r = 0; r < h; ++r) {
                        const float keep = upper ? d[r + h] : d[r], give = upper ? d[r] : d[r + h];
                        d[r] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                }
#pragma unroll
                for (int o = P / 2; o > 0; o >>= 1) d[0] += __shfl_xor_sync(0xffffffffu, d[0], o);
                if ((lane & (P - 1)) == 0) red[g][i & 1][(lane / P) * W + warp] = d[0];
            };
            // stage i: y of its rows, and y times the rows into p's sums
            auto second_half = [&](int i, const Quad (&w)[R][V], const float (&u)[R]) {
                const int st = st0 + i * st_step, cnt = min(R, rows - st * R);
                const int part_l = lane & (P - 1);
                float t = 0.0f;
                if (part_l * NV < W) {
                    const float* src = &red[g][i & 1][(lane / P) * W + part_l * NV];
#pragma unroll
                    for (int e = 0; e < NV; ++e) t += src[e];
                }
#pragma unroll
                for (int o = P / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                t = lane / P < cnt ? t * inv_v : 0.0f;
                if (k == p.it && warp == 0 && part_l == 0 && lane / P < cnt) p.y[row0 + st * R + lane / P] = t;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float yr = __shfl_sync(0xffffffffu, t, r * P);
                    sqsum = fmaf(yr, yr, sqsum);
                    if (has_rank) uy = fmaf(yr, u[r], uy);
                    const unsigned long long yy = pair(yr, yr);
#pragma unroll
                    for (int c = 0; c < V; ++c) {
                        pacc[c].lo = pair_fma(yy, w[r][c].lo, pacc[c].lo);
                        pacc[c].hi = pair_fma(yy, w[r][c].hi, pacc[c].hi);
                    }
                }
            };
            // the group is past the loads of one more stage: its slot takes the next copy
            auto stage_read = [&]() {
                group_sync(1 + g, TR);
                if (tg == 0 && q + p.slots < n_loads) issue();
                ++q;
                if (!p.resident && ++slot == p.slots) {
                    slot = 0;
                    parity ^= 1u;
                }
            };
            Quad wa[R][V], wb[R][V];
            float ua[R], ub[R];
            if (SG > 0) {
                first_half(0, wa, ua);
                first_sums(0, wa, ua);
                stage_read();
            }
            for (int i = 0; i < SG; i += 2) {
                if (i + 1 < SG) {
                    first_half(i + 1, wb, ub);
                    second_half(i, wa, ua);
                    first_sums(i + 1, wb, ub);
                    stage_read();
                } else {
                    second_half(i, wa, ua);
                    break;
                }
                if (i + 2 < SG) {
                    first_half(i + 2, wa, ua);
                    second_half(i + 1, wb, ub);
                    first_sums(i + 2, wa, ua);
                    stage_read();
                } else {
                    second_half(i + 1, wb, ub);
                }
            }
            back = !back;

            // ---- partial sums of the groups and of the CTA ----
            if constexpr (G > 1) {
                if (g > 0)
#pragma unroll
                    for (int c = 0; c < V; ++c)
                        *reinterpret_cast<ulonglong2*>(gsum + ((g - 1) * V + c) * TR + tg) = make_ulonglong2(pacc[c].lo, pacc[c].hi);
                __syncthreads();
            }
            if (g == 0) {
#pragma unroll
                for (int c = 0; c < V; ++c) {
                    float4 t;
                    asm("mov.b64 {%0, %1}, %2;" : "=f"(t.x), "=f"(t.y) : "l"(pacc[c].lo));
                    asm("mov.b64 {%0, %1}, %2;" : "=f"(t.z), "=f"(t.w) : "l"(pacc[c].hi));
#pragma unroll
                    for (int h = 0; h < G - 1; ++h) axpy(t, 1.0f, gsum[(h * V + c) * TR + tg]);
                    if (c * TR + tg < n4) __stcg(reinterpret_cast<float4*>(p.partial + (size_t)cta * n) + c * TR + tg, t);
                }
            }
            if (tg == 0) part[g][0] = sqsum;
            if (tg < j) part[g][1 + tg] = uy;
            __syncthreads();
            if (tid <= j) {
                float t = 0.0f;
#pragma unroll
                for (int h = 0; h < G; ++h) t += part[h][tid];
                __stcg(p.ext_rows + (size_t)tid * ctas + cta, t);
            }
            if (!grid_sync()) goto leave;

            // ---- this CTA's columns: p = (s (sum of the partial sums) - sum_l sigma_l (u_l y) v_l) / |y| ----
            for (int cb = c0; cb == c0 || cb < c1; cb += 8) {
                const int cl = tid & 7, run = tid >> 3, col = cb + cl;
                float4 t[kMaxCtas / 64], acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int e = 0; e < kMaxCtas / 64; ++e)
                    t[e] = col < c1 && run + 64 * e < ctas
                               ? __ldcg(reinterpret_cast<const float4*>(p.partial + (size_t)(run + 64 * e) * n) + col)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
                // what the last step needs, asked for now: v_l of the first ranks and the scale of its column
                constexpr int kAhead = 2;
                float4 vpre[kAhead], fpre = make_float4(1.f, 1.f, 1.f, 1.f);
                if (tid < 64 && cb + (tid >> 3) < c1) {
                    const int pc = cb + (tid >> 3);
#pragma unroll
                    for (int e = 0; e < kAhead; ++e)
                        if ((tid & 7) + 8 * e < j) vpre[e] = reinterpret_cast<const float4*>(p.V + (size_t)((tid & 7) + 8 * e) * n)[pc];
                    if (p.s != nullptr || p.s16 != nullptr) fpre = scale_of(p, pc);
                }
                if (cb == c0) {
                    for (int l = wid; l <= j; l += kWarps) {
                        const float x = cta_sum(p.ext_rows + (size_t)l * ctas, ctas, lane);
                        if (lane == 0) {
                            if (l == 0) s_yy = x;
                            else coef[l - 1] = sig[l - 1] * x;
                        }
                    }
                }
#pragma unroll
                for (int e = 0; e < kMaxCtas / 64; ++e) axpy(acc, 1.0f, t[e]);
                colred[run][cl] = acc;
                __syncthreads();
                if (tid < 64) {   // eight threads per column, each eight runs and every eighth rank, then three shuffles
                    const int cc = tid >> 3, e8 = tid & 7, pc = cb + cc;
                    float4 a = colred[e8][cc];
#pragma unroll
                    for (int e = 1; e < 8; ++e) axpy(a, 1.0f, colred[e8 + 8 * e][cc]);
                    if (pc < c1) {
                        a = make_float4(a.x * fpre.x, a.y * fpre.y, a.z * fpre.z, a.w * fpre.w);
#pragma unroll
                        for (int e = 0; e < kAhead; ++e)
                            if (e8 + 8 * e < j) axpy(a, -coef[e8 + 8 * e], vpre[e]);
                        for (int l = e8 + 8 * kAhead; l < j; l += 8)
                            axpy(a, -coef[l], reinterpret_cast<const float4*>(p.V + (size_t)l * n)[pc]);
                    }
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
                        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
                        a.z += __shfl_xor_sync(0xffffffffu, a.z, o);
                        a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
                    }
                    if (e8 == 0 && pc < c1) {
                        const float4 o = cast4(a, inv_norm(s_yy), 0);
                        __stcg(reinterpret_cast<float4*>(p.p) + pc, o);
                        own[pc - c0] = o;
                    }
                }
                __syncthreads();
            }
            for (int l = wid; l <= j; l += kWarps) {   // |p|^2 and v_l p over these columns
                float t = 0.0f;
                const float* po = reinterpret_cast<const float*>(own);
                const float* x = l == 0 ? po : p.V + (size_t)(l - 1) * n + 4 * c0;
                for (int e = lane; e < 4 * (c1 - c0); e += 32) t = fmaf(x[e], po[e], t);
                t = warp_sum(t);
                if (lane == 0) __stcg(p.ext_cols + (size_t)l * ctas + cta, t);
            }
            if (!grid_sync()) goto leave;
        }
        // ---- rank j is done: U[:, j] = y / |y|, V[j, :] = p / |p| (fp8 values when asked), sigma_j = |p| ----
        if (wid == 0) {
            const float t = cta_sum(p.ext_cols, ctas, lane);
            if (lane == 0) s_vv = t;
        }
        __syncthreads();
        const float iy = inv_norm(s_yy);
        ip = inv_norm(s_vv);
        rank_dead = iy == 0.0f || ip == 0.0f;   // exhausted, or something not finite: a zero triple
        const float sigma = rank_dead ? 0.0f : sqrtf(s_vv);
        for (int c = tid; c < c1 - c0; c += kThreads)
            reinterpret_cast<float4*>(p.V + (size_t)j * n)[c0 + c] =
                rank_dead ? make_float4(0.f, 0.f, 0.f, 0.f) : cast4(own[c], ip, p.cast);
        for (int i = tid; i < rows; i += kThreads) {
            float u = rank_dead ? 0.0f : p.y[row0 + i] * iy;
            if (p.cast) u = round_e4m3(u);
            p.U[(size_t)(row0 + i) * p.r + j] = u;
        }
        if (tid == 0) {
            sig[j] = sigma;
            if (cta == 0) p.sigma[j] = sigma;
        }
        __syncthreads();
    }
leave:
    // no copy may be in flight when the CTA leaves: after an aborted barrier, wait for those of this group
    if (s_abort) {
        if (tg == 0)
            for (int x = q; x < min(q + p.slots, n_loads); ++x)
                (void)mbar_wait(bar0 + 8u * (uint32_t)(x % p.slots), (uint32_t)(x / p.slots) & 1u);
        if (tid == 0) atomicExch(p.status, (int)LOPRO_ERR_TIMEOUT);
    }
}

// W <- W - sum_l sigma_l u_l v_l^T, ranks in ascending order: four rows per CTA share each piece of V.  Nothing if the
// sketch gave up (*status).
__global__ void __launch_bounds__(256) deflate_kernel(float* __restrict__ W, int m, int n, int r, const float* __restrict__ U,
                                                      const float* __restrict__ sigma, const float* __restrict__ V,
                                                      const int* __restrict__ status) {
    if (*status != (int)LOPRO_OK) return;
    constexpr int R = 4;
    const int i0 = blockIdx.x * R, live = min(R, m - i0), c4 = blockIdx.y * 256 + threadIdx.x;
    if (c4 >= n / 4) return;
    float4 a[R];
#pragma unroll
    for (int e = 0; e < R; ++e)
        if (e < live) a[e] = reinterpret_cast<const float4*>(W + (size_t)(i0 + e) * n)[c4];
    for (int l = 0; l < r; ++l) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(V + (size_t)l * n) + c4);
        const float sg = -__ldg(sigma + l);
#pragma unroll
        for (int e = 0; e < R; ++e)
            if (e < live) axpy(a[e], sg * __ldg(U + (size_t)(i0 + e) * r + l), v);
    }
#pragma unroll
    for (int e = 0; e < R; ++e)
        if (e < live) reinterpret_cast<float4*>(W + (size_t)(i0 + e) * n)[c4] = a[e];
}

template <int TR, int V, int R>
cudaError_t launch(SketchParams p, cudaStream_t s) {
    constexpr int G = kThreads / TR;
    static unsigned long long attr_done = 0;
    cudaError_t e = ensure_dynamic_smem(sketch_kernel<TR, V, R>, kRingBytes, &attr_done);
    if (e != cudaSuccess) return e;
    const int ctas = sm_count();
    const size_t stage = (size_t)R * p.n * 4;
    long long slots = (long long)kRingBytes / G / (long long)stage;
    if (slots > kMaxSlots / G) slots = kMaxSlots / G;
    const int rows = (p.m + ctas - 1) / ctas, stages = ((rows + R - 1) / R + G - 1) / G;
    p.slots = (int)slots;
    p.resident = stages <= slots;
    e = cudaMemsetAsync(p.sync - 2, 0, 16, s);  // the status word of the scratch with them
    if (e != cudaSuccess) return e;
    void* args[] = {&p};
    return cudaLaunchCooperativeKernel(sketch_kernel<TR, V, R>, dim3(ctas), dim3(kThreads), args, (size_t)kRingBytes, s);
}

}  // namespace

bool sketch_supported(int n, int r) {
    const int ctas = sm_count();
    return n <= 12288 && r <= kMaxRank && ctas <= kMaxCtas && (n / 4 + ctas - 1) / ctas <= kMaxOwn;
}

size_t sketch_scratch_bytes(int m, int n, int r) {
    const size_t ctas = (size_t)sm_count();
    return round_up_size(ctas * n * 4, 256) + 2 * round_up_size(ctas * (1 + (size_t)r) * 4, 256) +
           round_up_size((size_t)m * 4, 256) + round_up_size((size_t)n * 4, 256) + 256;
}

// All 512 threads share a row from 1025 columns on; rows per stage: what eight float4 of registers hold (they are held
// twice).  Up to 12288 columns (six float4).
cudaError_t launch_sketch(const SketchJob& job, void* scratch, cudaStream_t s) {
    SketchParams p = {};
    p.w = job.w;
    p.sketches = job.sketches;
    p.s = job.s;
    p.s_eff = job.s_eff;
    p.s16 = job.s16;
    p.U = job.U;
    p.sigma = job.sigma;
    p.V = job.V;
    p.status = job.status;
    p.m = job.m;
    p.n = job.n;
    p.r = job.r;
    p.it = job.it;
    p.cast = job.cast;
    uint8_t* b = (uint8_t*)scratch;
    auto take = [&](size_t bytes) {
        uint8_t* at = b;
        b += round_up_size(bytes, 256);
        return at;
    };
    const size_t ctas = (size_t)sm_count();
    p.sync = (unsigned*)take(256) + 2;  // (sketch_status in front)
    p.partial = (float*)take(ctas * p.n * 4);
    p.ext_rows = (float*)take(ctas * (1 + (size_t)p.r) * 4);
    p.ext_cols = (float*)take(ctas * (1 + (size_t)p.r) * 4);
    p.y = (float*)take((size_t)p.m * 4);
    p.p = (float*)take((size_t)p.n * 4);
    if (p.n <= 512) return launch<128, 1, 8>(p, s);
    if (p.n <= 1024) return launch<256, 1, 8>(p, s);
    if (p.n <= 2048) return launch<512, 1, 8>(p, s);
    if (p.n <= 4096) return launch<512, 2, 4>(p, s);
    if (p.n <= 8192) return launch<512, 4, 2>(p, s);
    return launch<512, 6, 1>(p, s);
}

cudaError_t launch_deflate(float* w, int m, int n, int r, const float* U, const float* sigma, const float* V, const int* status,
                           cudaStream_t s) {
    deflate_kernel<<<dim3((m + 3) / 4, (n / 4 + 255) / 256), 256, 0, s>>>(w, m, n, r, U, sigma, V, status);
    return cudaGetLastError();
}

}  // namespace lopro
