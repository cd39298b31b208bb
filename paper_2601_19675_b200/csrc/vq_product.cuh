// Product of the vector-quantized forward: y += W^_vq x~ for up to 32 token rows, W^ looked up centroid by centroid.
//
// What bounds it: shared-memory reads.  A 16 x 64 tile is 256 lookups of 8 bytes (4-D) at data-dependent addresses; with
// one copy of a codebook in shared memory the sixteen lanes of a half-warp hit sixteen random bank pairs and a read takes
// four to six passes instead of two, and every 16-row CTA copied all codebooks of its row group again.  Here
//  * a codebook is EXPANDED in shared memory: every lane position of a half-warp has a copy of its own in its own banks
//    (16 copies of 8 bytes per entry, 32 KB; 8 copies where a stage touches more than two codebooks; 32 copies of 4 bytes
//    for 2-D centroids), so that a lookup never conflicts; an entry's copies are 128 bytes, its address is the shifted and
//    masked index OR the lane's place: two instructions;
//  * a CTA works on a whole row block (up to 512 rows that share codebooks) one stage of 256 columns at a time: a codebook
//    is expanded once per block, and two 16-row tiles of a warp share every activation fragment;
//  * the stages of all row blocks are one list, cut evenly over one CTA per multiprocessor; a CTA leaves one partial sum
//    per row block that it touches, and a second launch adds them in order, with the low-rank term.
// A lane of a warp (row g, lane position t) takes the columns 64 t .. 64 t + 63 of a stage -- its indices are 16
// consecutive bytes (24 for 2-D) --, product j of the stage stands for its columns 64 t + 4 j .. + 3; the activation
// fragments follow the same assignment.  K phases: where a block has fewer than 32 tiles, PH groups of warps share the
// sixteen products of a stage.
// 8192 -> 28672, codebooks of 512 x 256, whole forward: 4 tokens 91.9 -> 42.8 us, 16 tokens 129.7 -> 55.7; with 2-D centroids
// 1 token 90.5 -> 52.2.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace lopro {

constexpr int kVqThreads = 512;
constexpr int kVqExpandedAt = 32768;   // shared-memory address of the expanded codebooks: above the raw ones, aligned so
                                       // that indices can be OR-ed in

enum { kVqDim4 = 0, kVqDim4Half = 1, kVqDim2 = 2 };  // 16 copies, 8 copies, 2-D
__host__ __device__ constexpr int vq_slot_bytes(int kind) { return kind == kVqDim4 ? 32768 : (kind == kVqDim4Half ? 16384 : 8192); }
__host__ __device__ constexpr int vq_raw_bytes(int kind) { return kind == kVqDim2 ? 256 : 2048; }

struct VqProduct {
    const uint8_t* idx;
    const unsigned char* books;
    const unsigned char* x;     // rotated activations of the launch's tokens: (col >> 10) * x_stage + token * x_token + 2 (col & 1023)
    int64_t x_stage, x_token;
    float* partial;             // [segment][phase][group of 4 tokens][row of the block][4]
    int m, n, T, cb_rows, cb_cols, n_cg;
    int max_books;              // codebooks that a stage touches, at most
    int stages;                 // per row block
    int total;                  // stages of all row blocks
    int ctas;
    uint32_t inv_stages, inv_cb_cols, inv_group;  // reciprocals for vq_div
};

// q / d by the host's reciprocal ceil(2^32 / d) (0 for d = 1): exact for q d < 2^32, which q < 2^20 stages of at most 128 per
// block, columns below 2^15 and fewer than 2^14 row blocks keep.  (Plain divisions cost
// 5 us of 48 on the 8192 -> 28672 layer.)
inline uint32_t vq_reciprocal(int d) { return d <= 1 ? 0u : (uint32_t)(((1ull << 32) + (uint32_t)d - 1) / (uint32_t)d); }
__device__ __forceinline__ int vq_div(int q, uint32_t inv) { return inv == 0u ? q : (int)__umulhi((uint32_t)q, inv); }

__host__ __device__ inline int vq_first_stage(int total, int ctas, int c) { return (int)((long long)total * c / ctas); }

template <int NT, int PH, int KIND>
__global__ void __launch_bounds__(kVqThreads, 1) vq_product_kernel(const VqProduct p) {
    constexpr int PAIRS = 16 / PH, RB = PAIRS * 32;
    constexpr int SLOT = vq_slot_bytes(KIND), RAW = vq_raw_bytes(KIND);
    constexpr int NW = (KIND == kVqDim2 ? 6 : 4) / PH;       // index words of a lane, row and stage
    constexpr int XS = NT * 4096;                            // activations of a stage
    extern __shared__ __align__(16) unsigned char vq_dyn[];
    __shared__ __align__(16) unsigned char zero_s[128];      // what the lanes beyond the last column look up
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int pair = warp % PAIRS, ph = warp / PAIRS;
    const uint32_t raw = smem_u32(vq_dyn), x_s = kVqExpandedAt + 2u * (uint32_t)p.max_books * SLOT;
    const int q0 = vq_first_stage(p.total, p.ctas, (int)blockIdx.x), q1 = vq_first_stage(p.total, p.ctas, (int)blockIdx.x + 1);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid < 8) reinterpret_cast<uint4*>(zero_s)[tid] = make_uint4(0, 0, 0, 0);

    auto cp16 = [](uint32_t dst, const void* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); };
    struct Place {
        int block, s, rg, fb, books;
    };
    auto place = [&](int q) {
        Place a;
        a.block = vq_div(q, p.inv_stages);
        a.s = q - a.block * p.stages;
        a.rg = vq_div(a.block, p.inv_group);
        a.fb = vq_div(a.s * 256, p.inv_cb_cols);
        a.books = vq_div(min(a.s * 256 + 256, p.n) - 1, p.inv_cb_cols) - a.fb + 1;
        return a;
    };
    auto load_books = [&](int q, const Place& a) {
        if (tid * 16 < a.books * RAW)
            cp16(raw + (uint32_t)((q & 1) * p.max_books * RAW + tid * 16), p.books + ((size_t)a.rg * p.n_cg + a.fb) * RAW + tid * 16);
    };
    auto load_x = [&](int s, int slot) {
        const uint32_t dst = x_s + (uint32_t)slot * XS;
        for (int i = tid; i < NT * 256; i += kVqThreads) {
            const int tok = i >> 5, c = i & 31, col = s * 256 + 8 * c;
            const bool on = tok < p.T && col < p.n;
            const unsigned char* src = on ? p.x + (size_t)(col >> 10) * p.x_stage + (size_t)tok * p.x_token + 2 * (col & 1023) : p.x;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)((((tok >> 3) * 8 + (c & 7)) * 32 +
                             (tok & 7) * 4 + (c >> 3)) * 16)), "l"(src), "r"(on ? 16 : 0) : "memory");
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    // codebooks of stage q into the buffer of its parity
    auto expand = [&](int q, int books) {
        for (int k = 0; k < books; ++k) {
            const uint32_t src = raw + (uint32_t)((q & 1) * p.max_books + k) * RAW;
            const uint32_t dst = kVqExpandedAt + (uint32_t)((q & 1) * p.max_books + k) * SLOT;
            if constexpr (KIND == kVqDim2) {
                const int e = warp * 4 + (lane >> 3);
                uint32_t v;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(src + 4u * (uint32_t)e) : "memory");
                asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(dst + (uint32_t)(e * 128 + (lane & 7) * 16)), "r"(v) : "memory");
            } else {
                constexpr int PER = KIND == kVqDim4 ? 8 : 4;   // lanes that write an entry's copies
#pragma unroll
                for (int e0 = 0; e0 < 256; e0 += 16 * 32 / PER) {
                    const int e = e0 + warp * (32 / PER) + lane / PER;
                    uint32_t a, b;
                    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(a), "=r"(b) : "r"(src + 8u * (uint32_t)e) : "memory");
                    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%1,%2};" ::"r"(dst + (uint32_t)(e * 16 * PER + (lane % PER) * 16)), "r"(a), "r"(b) : "memory");
                }
            }
        }
    };
    const size_t row_bytes = KIND == kVqDim2 ? (size_t)(p.n / 8 * 3) : (size_t)(p.n / 4);
    constexpr int kStageIdx = KIND == kVqDim2 ? 96 : 64;
    // the lane's index words of stage q: rows g, g + 8 of the warp's two tiles
    auto load_idx = [&](uint32_t (&w)[4][NW], int q, const Place& a) {
        const int row = a.block * RB + pair * 32 + g;
        const bool on = q < q1 && row < p.m && a.s * 256 + 64 * t < p.n;
        const uint8_t* src = p.idx + (size_t)row * row_bytes + (size_t)(a.s * kStageIdx + t * (kStageIdx / 4) + ph * (kStageIdx / 4 / PH));
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint8_t* rp = src + (size_t)(8 * r) * row_bytes;
            if constexpr (KIND != kVqDim2 && PH == 1) {
                const uint4 v = on ? __ldcs(reinterpret_cast<const uint4*>(rp)) : make_uint4(0, 0, 0, 0);
                w[r][0] = v.x; w[r][1] = v.y; w[r][2] = v.z; w[r][3] = v.w;
            } else if constexpr ((KIND != kVqDim2 && PH == 2) || (KIND == kVqDim2 && PH == 1)) {
#pragma unroll
                for (int e = 0; e < NW / 2; ++e) {
                    const uint2 v = on ? __ldcs(reinterpret_cast<const uint2*>(rp) + e) : make_uint2(0, 0);
                    w[r][2 * e] = v.x;
                    w[r][2 * e + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int e = 0; e < NW; ++e) w[r][e] = on ? __ldcs(reinterpret_cast<const uint32_t*>(rp) + e) : 0u;
            }
        }
    };

    float acc[2][NT][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][nt][e] = 0.0f;

    // centroid(s) of product jj (of this phase) for the row of w: the operand's two registers
    auto lookup = [&](const uint32_t (&w)[NW], int jj, uint32_t base, uint32_t& a_lo, uint32_t& a_hi) {
        if constexpr (KIND == kVqDim2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int bit = 6 * (2 * jj + h), word = bit >> 5, off = bit & 31;
                uint32_t v;
                if (off > 26) v = __funnelshift_r(w[word], w[word + 1 < NW ? word + 1 : word], off - 7);
                else v = off >= 7 ? w[word] >> (off >= 7 ? off - 7 : 0) : w[word] << (off < 7 ? 7 - off : 0);
                v = (v & 0x1F80u) | base;
                uint32_t& a = h ? a_hi : a_lo;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a) : "r"(v));
            }
        } else {
            constexpr int LG = KIND == kVqDim4 ? 7 : 6;        // an entry's copies are 2^LG bytes
            const int word = jj >> 2, sh = 8 * (jj & 3) - LG;
            const uint32_t v = sh >= 0 ? w[word] >> (sh >= 0 ? sh : 0) : w[word] << (sh < 0 ? -sh : 0);
            asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(a_lo), "=r"(a_hi) : "r"((v & (255u << LG)) | base));
        }
    };

    uint32_t cur[4][NW], nxt[4][NW];
    Place a = place(q0), a1 = place(q0 + 1), a2;   // this stage, the next, the one after
    int slot = 0;                                  // of this stage's activations
    if (q0 < q1) {
        load_books(q0, a);
        load_idx(cur, q0, a);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (q0 < q1) load_x(a.s, 0);
    commit();
    if (q0 + 1 < q1) {
        load_books(q0 + 1, a1);
        load_x(a1.s, 1);
    }
    commit();
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (q0 < q1) expand(q0, a.books);

    for (int q = q0; q < q1; ++q) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // stage q + 1
        __syncthreads();                                       // ... for every warp; stage q is expanded, stage q - 1 done with
        a2 = place(q + 2);
        if (q + 2 < q1) {
            load_books(q + 2, a2);
            load_x(a2.s, slot == 0 ? 2 : slot - 1);            // (slot + 2) mod 3
        }
        commit();
        load_idx(nxt, q + 1, a1);
        if (q + 1 < q1) expand(q + 1, a1.books);
        const int col = a.s * 256 + 64 * t;
        uint32_t base = smem_u32(zero_s);                      // (the indices of such a lane are 0)
        if (col < p.n)
            base = kVqExpandedAt + (uint32_t)((q & 1) * p.max_books + (vq_div(col, p.inv_cb_cols) - a.fb)) * SLOT +
                   (KIND == kVqDim2 ? (uint32_t)lane * 4u : (uint32_t)(lane & (KIND == kVqDim4 ? 15 : 7)) * 8u);
        const int row0 = a.block * RB + pair * 32;
        const uint32_t xs = x_s + (uint32_t)slot * XS + (uint32_t)(ph * (8 / PH) * 512 + lane * 16);
        if (row0 < p.m) {
#pragma unroll
            for (int qq = 0; qq < 8 / PH; ++qq) {
                uint32_t fa[2][2][4];   // [product][tile]
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        lookup(cur[2 * i], 2 * qq + h, base, fa[h][i][0], fa[h][i][2]);
                        lookup(cur[2 * i + 1], 2 * qq + h, base, fa[h][i][1], fa[h][i][3]);
                    }
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    uint4 b;
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "r"(xs + (uint32_t)((nt * 8 + qq) * 512)));
#pragma unroll
                    for (int i = 0; i < 2; ++i) mma_bf16(acc[i][nt], fa[0][i], b.x, b.y);
#pragma unroll
                    for (int i = 0; i < 2; ++i) mma_bf16(acc[i][nt], fa[1][i], b.z, b.w);
                }
            }
        }
        if (a.s == p.stages - 1 || q == q1 - 1) {
            // the end of a row block or of the CTA's list: segment number CTA + block (each grows along the list)
            if (row0 < p.m) {
                float* dst = p.partial + (size_t)((int)blockIdx.x + a.block) * (NT * 8 * 512) + (size_t)ph * (NT * 2 * RB * 4) +
                             (size_t)((t >> 1) * RB + pair * 32 + g) * 4 + (t & 1) * 2;
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            __stcg(reinterpret_cast<float2*>(dst + (size_t)(nt * 2 * RB + i * 16 + h * 8) * 4),
                                   make_float2(acc[i][nt][2 * h], acc[i][nt][2 * h + 1]));
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[i][nt][e] = 0.0f;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int e = 0; e < NW; ++e) cur[r][e] = nxt[r][e];
        a = a1;
        a1 = a2;
        if (++slot == 3) slot = 0;
    }
}

// y[token][row] = sum of the row block's partial sums (CTAs and phases in order) + A[row] . t[token]; grid (rows / 128,
// groups of four tokens), one row per thread.
__global__ void __launch_bounds__(128) vq_finish_kernel(const VqProduct p, int groups, int rb, int phases, const __half* __restrict__ A,
                                                        const __half* __restrict__ tv, int r_pad, void* __restrict__ y, int64_t ldy,
                                                        int out_f32) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int row = blockIdx.x * 128 + threadIdx.x, tg = blockIdx.y;
    const int block = row / rb, row_l = row - block * rb, first = block * p.stages;
    int c = (int)((long long)first * p.ctas / p.total);
    while (c > 0 && vq_first_stage(p.total, p.ctas, c) > first) --c;
    while (vq_first_stage(p.total, p.ctas, c + 1) <= first) ++c;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (row >= p.m) return;
    int end = c;
    while (end < p.ctas && vq_first_stage(p.total, p.ctas, end) < first + p.stages) ++end;
    // (segment, phase) in order, eight in flight: a narrow layer has its few row blocks cut into many segments
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4* src = reinterpret_cast<const float4*>(p.partial) + (size_t)(c + block) * ((size_t)groups * 512) + (size_t)tg * rb + row_l;
    const int count = (end - c) * phases;
    for (int k0 = 0; k0 < count; k0 += 8) {
        float4 a[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)   // groups * rb float4 per phase, groups * 512 per segment = phases of them
            a[k] = k0 + k < count ? __ldcg(src + (size_t)(k0 + k) * ((size_t)groups * rb)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v.x += a[k].x;
            v.y += a[k].y;
            v.z += a[k].z;
            v.w += a[k].w;
        }
    }
    float o[4] = {v.x, v.y, v.z, v.w};
    for (int j = 0; j < r_pad / 8; ++j) {
        const uint4 av = __ldg(reinterpret_cast<const uint4*>(A + (size_t)row * r_pad) + j);
        const __half2* ah = reinterpret_cast<const __half2*>(&av);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int tok = min(tg * 4 + e, p.T - 1);
            const uint4 bv = __ldcg(reinterpret_cast<const uint4*>(tv + (size_t)tok * r_pad) + j);
            const __half2* bh = reinterpret_cast<const __half2*>(&bv);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 fa = __half22float2(ah[q]), fb = __half22float2(bh[q]);
                o[e] = fmaf(fa.x, fb.x, o[e]);
                o[e] = fmaf(fa.y, fb.y, o[e]);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int tok = tg * 4 + e;
        if (tok >= p.T) break;
        if (out_f32) reinterpret_cast<float*>(y)[(size_t)tok * ldy + row] = o[e];
        else reinterpret_cast<__nv_bfloat16*>(y)[(size_t)tok * ldy + row] = __float2bfloat16_rn(o[e]);
    }
}

}  // namespace lopro
