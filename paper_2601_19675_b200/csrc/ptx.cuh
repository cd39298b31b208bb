// Device helpers shared by the small-batch kernels: mbarrier and bulk-copy wrappers with bounded
// waits, warp-level tensor-core instructions, and the expansion of packed codes into bf16 operands.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace lopro {

constexpr uint32_t kSpinLimit = 1u << 22;  // polls of one mbarrier wait before it gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// one poll that never suspends the thread
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// try_wait with a suspend-time hint (ns): the thread may stay parked that long before the instruction returns false
__device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar, uint32_t parity, uint32_t hint_ns) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(hint_ns)
        : "memory");
    return ok != 0;
}
// Bounded wait for warps that expect to wait long: a failed poll backs off before the next one, so that the polls
// of many waiting warps do not crowd the shared-memory pipeline of the warps that work.
__device__ __forceinline__ bool mbar_wait_backoff(uint32_t bar, uint32_t parity, uint32_t limit = kSpinLimit) {
    for (uint32_t i = 0; i < limit; ++i) {
#if defined(RB_WAIT_HINT)
        if (mbar_try_wait_hint(bar, parity, RB_WAIT_HINT)) return true;
#else
        if (mbar_try_wait(bar, parity)) return true;
#endif
#if defined(RB_WAIT_SLEEP)
        __nanosleep(RB_WAIT_SLEEP);
#endif
    }
    return false;
}
// Bounded wait: false if the limit ran out (the caller records the time-out and carries on).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit = kSpinLimit) {
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// First product of a chain: D = A B with a zero C operand (no registers to clear).
__device__ __forceinline__ void mma_bf16_first(float (&d)[4], const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// Loads from shared memory by 32-bit address, kept behind the waits in front of them.
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float lds_f32(uint32_t addr) { return __uint_as_float(lds32(addr)); }
// a lane's words of one tile step: one 16- or 8-byte load, three words one by one
template <int BITS>
__device__ __forceinline__ void lds_words(uint32_t (&w)[BITS], uint32_t addr) {
    if constexpr (BITS == 4) {
        asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(addr) : "memory");
    } else if constexpr (BITS == 2) {
        asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(addr) : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < BITS; ++q) w[q] = lds32(addr + 4u * q);
    }
}

// two fp8 e4m3 values (low byte first) -> two fp16 values (exact)
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint16_t v) {
    uint32_t d;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(d) : "h"(v));
    return d;
}

// A-operand registers (m16n8k16, fp16) of the 16 x 16 piece at columns jj of a 16-row tile of the up-projection
// factor held in shared memory, rows r_pad entries apart: fp16 entries (A = U Sigma), or fp8 e4m3 entries (U of the
// FP8 low-rank record) converted exactly to fp16.
__device__ __forceinline__ void load_up_fragment(uint32_t (&a)[4], const unsigned char* tile, int r_pad, int gq, int tg, int jj,
                                                 bool lr8) {
    if (!lr8) {
        const __half* as = reinterpret_cast<const __half*>(tile);
        a[0] = *reinterpret_cast<const uint32_t*>(as + gq * r_pad + jj + 2 * tg);
        a[1] = *reinterpret_cast<const uint32_t*>(as + (gq + 8) * r_pad + jj + 2 * tg);
        a[2] = *reinterpret_cast<const uint32_t*>(as + gq * r_pad + jj + 8 + 2 * tg);
        a[3] = *reinterpret_cast<const uint32_t*>(as + (gq + 8) * r_pad + jj + 8 + 2 * tg);
    } else {
        a[0] = e4m3x2_to_f16x2(*reinterpret_cast<const uint16_t*>(tile + gq * r_pad + jj + 2 * tg));
        a[1] = e4m3x2_to_f16x2(*reinterpret_cast<const uint16_t*>(tile + (gq + 8) * r_pad + jj + 2 * tg));
        a[2] = e4m3x2_to_f16x2(*reinterpret_cast<const uint16_t*>(tile + gq * r_pad + jj + 8 + 2 * tg));
        a[3] = e4m3x2_to_f16x2(*reinterpret_cast<const uint16_t*>(tile + (gq + 8) * r_pad + jj + 8 + 2 * tg));
    }
}

constexpr uint32_t kMagic128 = 0x43004300u;  // two bf16 128.0 (ulp 1): 128.0 | c == 128 + c

// (a & mask) | magic in ONE logic instruction (truth table 0xEA), both constants held in registers --
// left to the compiler this becomes two instructions, since only one operand may be an immediate.
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t mask, uint32_t magic) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(mask), "r"(magic));
    return d;
}

template <int BITS>
__device__ __forceinline__ void expand_codes(uint32_t (&a)[16], const uint32_t (&w)[BITS]) {
    const uint32_t magic = kMagic128;
    if constexpr (BITS == 4) {
        const uint32_t mask = 0x000F000Fu;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int rho = 0; rho < 4; ++rho) a[4 * j + rho] = and_or(w[j] >> (4 * rho), mask, magic);
    } else if constexpr (BITS == 2) {
        const uint32_t mask = 0x00030003u;
#pragma unroll
        for (int pi = 0; pi < 16; ++pi) a[pi] = and_or(w[pi >> 3] >> (2 * (pi & 7)), mask, magic);
    } else {
        const uint32_t mask = 0x00070007u;
#pragma unroll
        for (int pi = 0; pi < 15; ++pi) a[pi] = and_or(w[pi / 5] >> (3 * (pi % 5)), mask, magic);
        a[15] = ((w[0] >> 15) & 0x00010001u) | ((w[1] >> 14) & 0x00020002u) | ((w[2] >> 13) & 0x00040004u) | kMagic128;
    }
}

// The same with fewer shifts for the kernels that scale rows afterwards: the odd pairs, which are the rows gq + 8 of a tile,
// come out as 128 + kOdd c, their bits left where a shift that an even pair needs anyway puts them (2 bits: 6 shifts instead of
// 14 per tile step, 3 bits: 10 instead of 15).  kOdd is a power of two and comes off with the rows' scale, exactly.  The
// operands of those rows reach 140 (2 bits) and 184 (3 bits) instead of 131 and 135: the products of one step leave the fp32
// range where its 64 |x~| add up to 1.8e36 or more (2.5e36 with operands up to 135).  The loops these
// serve are bound by instruction issue with the integer pipe next; with the packed multiply-adds below, in the kernels that ran them
// then, 8192 -> 28672 at 2 bits, 16 tokens 51.4 -> 48.8 us (tall.cu), 11008 -> 4096 at 3 bits, 5 tokens 14.5 -> 14.0 (stream.cu).
template <int BITS>
struct OddRows {
    static constexpr float factor = BITS == 4 ? 1.0f : (BITS == 2 ? 4.0f : 8.0f);
};
template <int BITS>
__device__ __forceinline__ void expand_codes_by_rows(uint32_t (&a)[16], const uint32_t (&w)[BITS]) {
    const uint32_t magic = kMagic128;
    if constexpr (BITS == 4) {
        expand_codes<4>(a, w);
    } else if constexpr (BITS == 2) {
        // word h holds pairs 8h .. 8h + 7 at bits 2p: two pairs per shift by 4
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t v = w[h] >> (4 * k);
                a[8 * h + 2 * k] = and_or(v, 0x00030003u, magic);
                a[8 * h + 2 * k + 1] = and_or(v, 0x000C000Cu, magic);
            }
    } else {
        // words 0 and 2: even pairs at bits 0, 6, 12, odd ones at 3, 9; word 1: odd pairs at 0, 6, 12, even ones at 3, 9
        const uint32_t even = 0x00070007u, odd = 0x00380038u;
#pragma unroll
        for (int h = 0; h < 3; h += 2) {
            const uint32_t v = w[h] >> 6;
            a[5 * h] = and_or(w[h], even, magic);
            a[5 * h + 1] = and_or(w[h], odd, magic);
            a[5 * h + 2] = and_or(v, even, magic);
            a[5 * h + 3] = and_or(v, odd, magic);
            a[5 * h + 4] = and_or(w[h] >> 12, even, magic);
        }
        const uint32_t v3 = w[1] >> 3, v9 = w[1] >> 9;
        a[5] = and_or(w[1] << 3, odd, magic);
        a[6] = and_or(v3, even, magic);
        a[7] = and_or(v3, odd, magic);
        a[8] = and_or(v9, even, magic);
        a[9] = and_or(v9, odd, magic);
        // pair 15: bit b at bit 15 (and 31) of word b, wanted at bit 3 + b
        a[15] = and_or(w[2] >> 10, 0x00200020u, and_or(w[1] >> 11, 0x00100010u, and_or(w[0] >> 12, 0x00080008u, magic)));
    }
}

// The products of one step with NT token tiles, the tiles of a quarter step one after the other: products that follow each
// other then do not wait for one another (8192 -> 4096 at 4 bits, 24 tokens: 25.2 us tile by tile, 24.8 this way).
template <int NT>
__device__ __forceinline__ void multiply_step(float (&acc)[NT][4], const uint32_t (&a)[16], const uint32_t (&b)[NT][8]) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) mma_bf16_first(acc[nt], &a[0], b[nt][0], b[nt][1]);
#pragma unroll
    for (int k = 1; k < 4; ++k)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma_bf16(acc[nt], &a[4 * k], b[nt][2 * k], b[nt][2 * k + 1]);
}

// Two fp32 multiply-adds in one issue slot; the halves of a register pair are two tokens of a row.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Scale and zero-point of a group for the rows gq (.x) and gq + 8 (.y) of a tile, as the sums of a tile step meet them:
// y += s (acc - (128 + z) sum x~); for the odd rows acc = sum (128 + kOdd c) x~, and s and z are those of kOdd c.
template <int BITS>
struct RowScales {
    float s[2], z[2];
    __device__ __forceinline__ RowScales(uint32_t sz_lo, uint32_t sz_hi) {
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&sz_lo));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&sz_hi));
        s[0] = lo.x;
        s[1] = hi.x * (1.0f / OddRows<BITS>::factor);
        z[0] = -128.0f - lo.y;
        z[1] = fmaf(hi.y, -OddRows<BITS>::factor, -128.0f);
    }
};
// Adds the products of one step to the sums of a tile: acc and y in the accumulator layout of m16n8k16 (rows gq, gq + 8,
// tokens 2 tg and 2 tg + 1 of NT token tiles), sx the step's column sums of those tokens.
template <int BITS, int NT>
__device__ __forceinline__ void add_scaled(float (&y)[NT][4], const float (&acc)[NT][4], const float (&sx)[NT][2], const RowScales<BITS>& r) {
    if constexpr (NT == 1) {   // (packed operands would cost the registers' copies that they save)
#pragma unroll
        for (int i = 0; i < 4; ++i) y[0][i] = fmaf(r.s[i >> 1], fmaf(r.z[i >> 1], sx[0][i & 1], acc[0][i]), y[0][i]);
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned long long s2 = pack2(r.s[h], r.s[h]), z2 = pack2(r.z[h], r.z[h]);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const unsigned long long t = fma2(z2, pack2(sx[nt][0], sx[nt][1]), pack2(acc[nt][2 * h], acc[nt][2 * h + 1]));
                unpack2(fma2(s2, t, pack2(y[nt][2 * h], y[nt][2 * h + 1])), y[nt][2 * h], y[nt][2 * h + 1]);
            }
        }
    }
}

}  // namespace lopro
