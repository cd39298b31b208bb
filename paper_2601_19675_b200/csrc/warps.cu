// Small-batch forward (decode, T <= 32) with every warp on a run of its own: y = W^ x~ + A t  (steps "Dequant(W_q) X" and
// "U (Sigma Y)" of Appendix A.3, summed as in Eq. 8), after the prologue kernel that writes the rotated activations x~ (as the
// stage image), their 64-column sums and t = B x.
//
// One CTA per SM owns a contiguous run of 16-row tiles (the runs differ by at most one).  The tile steps of the run -- 16 rows x 64
// columns, tile by tile -- are cut into sixteen equal pieces, one per warp.  In the fragment layout the codes of neighbouring tile
// steps are neighbours in memory, and so are their (scale, zero) pairs: a warp's piece is one contiguous stream of each, which it
// fetches itself with 16-byte asynchronous copies, D batches of PER steps ahead, into a ring that no other warp reads.  Nothing in the
// loop waits for another warp.  (With one producer for all sixteen warps, as in the persistent kernel of tall.cu, a stage of 64 tile steps
// took some 2600 cycles however many bytes it held: nine bulk copies at 80 cycles of one thread each, between waits, on a scheduler
// shared with four busy warps; four producers or copies issued by the last warp of a stage were slower still.)  The activations of all of K are fetched once and stay.  A warp that leaves a tile, or ends, puts its
// sums of the tile into shared memory; when all are done, a warp per tile adds them in order, with the low-rank term.
//
// What bounds it: instruction issue with little to hide latency behind, four warps per scheduler.  Twice the integer instructions
// (expansion: two cycles per instruction and scheduler) plus eight times the products (m16n8k16 on the legacy tensor pipe), which share
// the way out of a scheduler, are what no loop over these operands gets below: 44 + 32 = 76 cycles per tile step at 2 bits and one token
// tile, 44 + 64 = 108 at two, 56 + 32 = 88 and 56 + 128 = 184 at 4 bits and one and four.  Instructions per step over the share of busy
// issue slots, way in and out included: 4096 -> 28672, 2 bits, 1 token 126 cycles (75 instructions, of which 49 are the step), eight
// experts 4096 -> 14336 97, 8192 -> 28672, 2 bits, 16 tokens 173, 4096 -> 11008, 4 bits, 8 tokens 202 (20 steps per warp), 32 tokens 408.
//
// Arithmetic as in stream.cu: sum_k s (c_k - z) x~_k = s (sum_k (128 + c_k) x~_k - (128 + z) sum_k x~_k),
// exact bf16 operands 128 + c_k on the tensor cores (rows gq + 8 of a tile: see expand_codes_by_rows), fp32 accumulation,
// scale and zero-point applied in fp32 once per 64 columns.
//
// Every mbarrier wait is bounded; a wait that runs out stores LOPRO_ERR_TIMEOUT in the workspace status word and the warp stops
// waiting (the outputs are then unspecified).
#include "common.cuh"
#include "ptx.cuh"

namespace lopro {

namespace {

constexpr int kWarps = 16;
constexpr int kMaxX = 32;   // stages of the activation image that a CTA may hold
constexpr int kRunMaxSmem = 226 * 1024;   // dynamic shared memory of a CTA

struct RunParams {
    const unsigned char* codes;
    const unsigned char* sz;
    const unsigned char* A;
    const unsigned char* act;  // activation image [stage][t_pad][kActRecord]
    const __half* t;           // [T][r_pad] low-rank intermediate
    int* status;
    void* y;
    int64_t ldy;
    int out_f32;
    int m, T, t_pad;
    int nsteps, gshift, r_pad;
    int lr8;       // the up-projection factor is fp8 e4m3 (U of the FP8 low-rank record), one byte per entry
    int n_clusters, cluster;   // units that the layers are shared out to: clusters of CTAs, each CTA a part of K
    // shared-memory layout (bytes from the dynamic base)
    int off_t, off_red, off_x, x_bytes, off_ring;
};

// Sibling layers of a grouped launch: the grid's clusters from cta0[i] on work on sibling i (the layer of RunParams
// owns those before cta0[0]); each sibling walks its own rows with its own share of the persistent CTAs.
struct RunSiblings {
    int n;
    int cta0[kMaxSiblings - 1];
    const unsigned char* codes[kMaxSiblings - 1];
    const unsigned char* sz[kMaxSiblings - 1];
    const unsigned char* A[kMaxSiblings - 1];
    const unsigned char* act[kMaxSiblings - 1];
    const __half* t[kMaxSiblings - 1];
    void* y[kMaxSiblings - 1];
    int64_t ldy[kMaxSiblings - 1];
    int m[kMaxSiblings - 1];
    int T[kMaxSiblings - 1];  // token rows of the sibling
};

// A launch of a single layer carries no table (several hundred bytes of kernel parameters less).
struct NoRunSiblings {};
__device__ __forceinline__ int2 select_sibling(RunParams& p, int unit, const NoRunSiblings&) { return make_int2(unit, p.n_clusters); }

// The layer that a cluster (a CTA where they are alone) works on: patches the per-layer fields, returns the cluster's index among
// the layer's and their number.
__device__ __forceinline__ int2 select_sibling(RunParams& p, int unit, const RunSiblings& sibs) {
    int idx = -1;
#pragma unroll
    for (int i = 0; i < kMaxSiblings - 1; ++i)
        if (i < sibs.n && unit >= sibs.cta0[i]) idx = i;
    if (idx < 0) return make_int2(unit, sibs.n > 0 ? sibs.cta0[0] : p.n_clusters);
    // (a __grid_constant__ parameter: one constant-bank load per field at a computed index)
    const int first = sibs.cta0[idx], end = idx + 1 < sibs.n ? sibs.cta0[idx + 1] : p.n_clusters;
    p.codes = sibs.codes[idx];
    p.sz = sibs.sz[idx];
    p.A = sibs.A[idx];
    p.act = sibs.act[idx];
    p.t = sibs.t[idx];
    p.y = sibs.y[idx];
    p.ldy = sibs.ldy[idx];
    p.m = sibs.m[idx];
    p.T = sibs.T[idx];
    return make_int2(unit - first, end - first);
}

__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// a piece of global memory (a multiple of 16 bytes) into L2
__device__ __forceinline__ void prefetch_l2(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// One 16-row tile times one 64-column step: the codes are expanded to bf16 operands 128 + c, multiplied (four m16n8k16 products
// per token tile), and scale and zero-point applied in fp32 against the step's column sums.
template <int BITS, int NT>
__device__ __forceinline__ void tile_step(uint32_t w_addr, uint32_t x_addr, uint32_t sz_addr, const float (&sx)[NT][2], float (&yacc)[NT][4]) {
    uint32_t w[BITS];
    lds_words<BITS>(w, w_addr);
    uint32_t b[NT][8];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        ldmatrix_x4(*reinterpret_cast<uint32_t(*)[4]>(&b[nt][0]), x_addr + (uint32_t)(nt * 8 * kActRecord));
        ldmatrix_x4(*reinterpret_cast<uint32_t(*)[4]>(&b[nt][4]), x_addr + (uint32_t)(nt * 8 * kActRecord + 64));
    }
    const uint32_t sz0 = lds32(sz_addr), sz1 = lds32(sz_addr + 32u);
    uint32_t a[16];
    expand_codes_by_rows<BITS>(a, w);
    float acc[NT][4];
    multiply_step<NT>(acc, a, b);
    add_scaled<BITS, NT>(yacc, acc, sx, RowScales<BITS>(sz0, sz1));
}

// Bytes of a ring slot: PER steps of codes, their (scale, zero) pairs.
template <int BITS, int PER>
__host__ __device__ constexpr int slot_bytes() {
    return PER * (128 * BITS + 64);
}

__device__ __forceinline__ float4 load_from_rank(uint32_t addr, uint32_t rank) {
    uint32_t there;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(there) : "memory");
    return v;
}
__device__ __forceinline__ float4 load_shared(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

// CLUSTER: the CTAs of a cluster share their tiles and take a part of K each (rank r of C the batches nb r / C .. nb (r + 1) / C of every
// tile), so that each holds its part of the activations only; at the end tile t is added up by rank t mod C.
template <int BITS, int NT, int PER, int D, bool CLUSTER>
__device__ __forceinline__ void run_body(const RunParams& p, const int2 cta) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[kMaxX + 1];  // full per stage of activations; t
    constexpr int kTok = NT * 8;
    constexpr int kStepBytes = 128 * BITS;               // codes of one 16-row tile and one 64-column step
    constexpr int kSlot = slot_bytes<BITS, PER>(), kBatch = PER * kStepBytes;
    static_assert(D * kSlot >= NT * 512, "a warp's last sums go where its ring was");

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gq = lane >> 2, tg = lane & 3;
    const int C = CLUSTER ? p.cluster : 1, rank = CLUSTER ? (int)blockIdx.x % C : 0;
    // this cluster's run of 16-row tiles: the first `extra` ones hold one tile more
    const int tiles = p.m >> 4;
    const int base = tiles / cta.y, extra = tiles - base * cta.y;
    const int my_cnt = base + (cta.x < extra ? 1 : 0);
    const int my_start = cta.x * base + min(cta.x, extra);
    // the warp's batches of PER tile steps, counted along the run; k0: the CTA's first step of a tile
    const int nb = p.nsteps / PER;
    const int k0 = CLUSTER ? nb * rank / C * PER : 0, per_tile = CLUSTER ? nb * (rank + 1) / C - nb * rank / C : nb, k1 = k0 + per_tile * PER, total = my_cnt * per_tile;
    const int stage0 = k0 >> 4, n_stages = ((k1 + 15) >> 4) - stage0;
    const int b0 = total * warp / kWarps, b1 = total * (warp + 1) / kWarps;
    const uint32_t bar0 = smem_u32(bars), smem0 = smem_u32(smem);
    const uint32_t tbar = bar0 + 8u * (uint32_t)kMaxX;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid < n_stages) mbar_init(bar0 + 8u * (uint32_t)tid, 1);
    if (tid == kMaxX) mbar_init(tbar, 1);
    if (tid <= kMaxX) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");

    // ---- the warp's ring ----
    const uint32_t ring0 = smem0 + (uint32_t)p.off_ring;
    const uint32_t ring = ring0 + (uint32_t)(warp * (D * kSlot)), ring_end = ring + D * kSlot;
    int tile = b0 / per_tile, k = k0 + (b0 - tile * per_tile) * PER;   // tile of the run, step of the tile
    int next = b0, pos = tile * p.nsteps + k, left = per_tile - (b0 - tile * per_tile);   // the next request: its batch, step of the run, batches to the tile's end
    const unsigned char* codes = p.codes + ((size_t)my_start * p.nsteps + pos) * kStepBytes + lane * 16;
    const unsigned char* sz = p.sz + (size_t)my_start * (size_t)(p.nsteps >> p.gshift) * 64 + lane * 16;
    uint32_t dst = ring + (uint32_t)lane * 16u;
    const bool sz_lane = lane < 4 * (PER >> min(p.gshift, PER == 4 ? 2 : 1));   // the pairs of PER steps: a group or more
    auto request = [&] {
        if (next < b1) {
#pragma unroll
            for (int q = 0; q < kBatch; q += 512)
                if (q + 512 <= kBatch || lane * 16 < kBatch - q) copy16(dst + (uint32_t)q, codes + q);
            if (sz_lane) copy16(dst + kBatch, sz + (uint32_t)((pos >> p.gshift) << 6));
            codes += kBatch;
            pos += PER;
            ++next;
            if (CLUSTER && --left == 0) {   // on to the next tile's part of K
                left = per_tile;
                pos += p.nsteps - (k1 - k0);
                codes += (p.nsteps - (k1 - k0)) * kStepBytes;
            }
            dst += kSlot;
            if (dst >= ring_end) dst -= D * kSlot;
        }
        copy_commit();
    };
    // (one batch of four steps: more of them held up the launch in front, 4096 -> 28672 at 4 tokens 16.9 and 17.9 us)
    constexpr int kEarly = NT == 4 ? D : 1;
#pragma unroll 1
    for (int q = 0; q < kEarly; ++q) request();
    const int t0 = rank + C * warp, t_step = C * kWarps;   // the tiles that this warp adds up at the end
    if (lane == 0 && p.r_pad > 0) {   // the rows of A, needed at the end, are on their way to L2
        const uint32_t tile_bytes = (uint32_t)(16 * p.r_pad * (p.lr8 ? 1 : 2));
        for (int tl = t0; tl < my_cnt; tl += t_step) prefetch_l2(p.A + (size_t)(my_start + tl) * tile_bytes, tile_bytes);
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (lane == 0 && my_cnt > 0) {
        const uint32_t bytes = (uint32_t)(min(kTok, p.T) * kActRecord);
        for (int q = warp; q < n_stages; q += kWarps) {
            mbar_expect_tx(bar0 + 8u * (uint32_t)q, bytes);
            bulk_g2s(smem0 + p.off_x + (uint32_t)(q * p.x_bytes), p.act + (size_t)(stage0 + q) * p.t_pad * kActRecord, bytes, bar0 + 8u * (uint32_t)q);
        }
        // low-rank intermediate of the live tokens, where this CTA adds up a tile: nobody else waits for it, and no CTA may leave with
        // a copy into its shared memory under way (a cluster with one tile: its second CTA adds up none)
        if (warp == kWarps - 1 && p.r_pad > 0 && rank < my_cnt) {
            const uint32_t t_bytes = (uint32_t)(min(kTok, p.T) * p.r_pad * 2);
            mbar_expect_tx(tbar, t_bytes);
            bulk_g2s(smem0 + p.off_t, p.t, t_bytes, tbar);
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int q = kEarly; q < D; ++q) request();

    bool dead = false;  // a wait of this warp ran out: it stops waiting
    auto wait = [&](uint32_t bar) {
        if (!dead && !mbar_wait(bar, 0)) {
            dead = true;
            if (lane == 0) atomicExch(p.status, (int)LOPRO_ERR_TIMEOUT);
        }
    };
    // Sums of a tile [token tile][lane] float4: a warp that goes on to the next tile leaves them in the slot of the tile that it ends
    // (one warp does, at most), a warp that is done where its ring was.
    auto put = [&](uint32_t to, const float (&v)[NT][4]) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
            asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(to + (uint32_t)((nt * 32 + lane) * 16)), "f"(v[nt][0]), "f"(v[nt][1]), "f"(v[nt][2]), "f"(v[nt][3]) : "memory");
    };
    // from a stage of activations: the lane's ldmatrix row, the column sums of token 2 tg
    const uint32_t x_ofs = smem0 + (uint32_t)(p.off_x + (lane & 7) * kActRecord + (lane >> 3) * 16 - stage0 * p.x_bytes);
    const uint32_t sx_ofs = smem0 + (uint32_t)(p.off_x + 2048 + 2 * tg * kActRecord - stage0 * p.x_bytes);
    // bytes from the (scale, zero) pairs of a slot's first step to those of the others
    const uint32_t g1 = p.gshift == 0 ? 64u : 0u, g2 = p.gshift == 0 ? 128u : (p.gshift == 1 ? 64u : 0u), g3 = p.gshift == 0 ? 192u : (p.gshift == 1 ? 64u : 0u);
    uint32_t src = ring;   // the slot that is consumed next
    float yacc[NT][4];
    if (b0 < b1) wait(bar0 + 8u * (uint32_t)((k >> 4) - stage0));
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) yacc[nt][i] = 0.0f;
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        copy_wait<D - 1>();
        __syncwarp();
        const uint32_t x0 = (uint32_t)((k >> 4) * p.x_bytes), kk = (uint32_t)(k & 15);
        const uint32_t w_addr = src + (uint32_t)(lane * (BITS * 4)), sz_addr = src + (uint32_t)(kBatch + gq * 4), x_addr = x_ofs + x0 + kk * 128u;
        float s4[NT][2][PER];   // column sums of the steps
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t a = sx_ofs + x0 + kk * 4u + (uint32_t)((nt * 8 + h) * kActRecord);
                if constexpr (PER == 4)
                    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                                 : "=f"(s4[nt][h][0]), "=f"(s4[nt][h][1]), "=f"(s4[nt][h][2]), "=f"(s4[nt][h][3]) : "r"(a) : "memory");
                else
                    asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(s4[nt][h][0]), "=f"(s4[nt][h][1]) : "r"(a) : "memory");
            }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            float sx[NT][2];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) sx[nt][h] = s4[nt][h][i];
            tile_step<BITS, NT>(w_addr + (uint32_t)(i * kStepBytes), x_addr + (uint32_t)(i * 128), sz_addr + (i == 0 ? 0u : (i == 1 ? g1 : (i == 2 ? g2 : g3))), sx, yacc);
        }
        src += kSlot;
        if (src == ring_end) src = ring;
        __syncwarp();
        request();
        k += PER;
        if (b == b1 - 1) break;
        if (k == k1) {
            put(smem0 + (uint32_t)(p.off_red + tile * (NT * 512)), yacc);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) yacc[nt][i] = 0.0f;
            k = k0;
            ++tile;
            if (k & 15) wait(bar0);
        }
        if ((k & 15) == 0) wait(bar0 + 8u * (uint32_t)((k >> 4) - stage0));
    }
    copy_wait<0>();
    __syncwarp();
    if (b0 < b1) put(ring, yacc);

    // ---- a warp per tile adds the warps' sums in order, with the low-rank term A t (fp16 tensor-core product), and stores the rows ----
    const int rp = p.r_pad, row_bytes = rp * (p.lr8 ? 1 : 2);
    auto load_a = [&](uint32_t (&a)[4], int tl, int jj) {
        const unsigned char* row = p.A + ((size_t)(my_start + tl) * 16 + gq) * row_bytes;
        if (!p.lr8) {
            const unsigned char* r0 = row + (jj + 2 * tg) * 2;
            a[0] = __ldg(reinterpret_cast<const uint32_t*>(r0));
            a[1] = __ldg(reinterpret_cast<const uint32_t*>(r0 + 8 * row_bytes));
            a[2] = __ldg(reinterpret_cast<const uint32_t*>(r0 + 16));
            a[3] = __ldg(reinterpret_cast<const uint32_t*>(r0 + 8 * row_bytes + 16));
        } else {
            const unsigned char* r0 = row + jj + 2 * tg;
            a[0] = e4m3x2_to_f16x2(__ldg(reinterpret_cast<const uint16_t*>(r0)));
            a[1] = e4m3x2_to_f16x2(__ldg(reinterpret_cast<const uint16_t*>(r0 + 8 * row_bytes)));
            a[2] = e4m3x2_to_f16x2(__ldg(reinterpret_cast<const uint16_t*>(r0 + 8)));
            a[3] = e4m3x2_to_f16x2(__ldg(reinterpret_cast<const uint16_t*>(r0 + 8 * row_bytes + 8)));
        }
    };
    uint32_t a0[4][4];   // the first tile's factor is on its way while the last warps finish
    if (t0 < my_cnt)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q * 16 < rp) load_a(a0[q], t0, q * 16);
    __syncthreads();
    // this CTA's sums of tile tl, warp by warp
    auto add_warps = [&](float (&sum)[NT][4], int tl) {
        const int first = tl * per_tile, last = first + per_tile - 1;
        int w = first * kWarps / total;
        while (w > 0 && total * w / kWarps > first) --w;
        while (total * (w + 1) / kWarps <= first) ++w;
#pragma unroll 1
        for (; w < kWarps && total * w / kWarps <= last; ++w) {
            const int end = total * (w + 1) / kWarps;
            if (total * w / kWarps == end) continue;   // (a warp without a batch)
            const uint32_t theirs = (end > last + 1 ? smem0 + (uint32_t)(p.off_red + tl * (NT * 512)) : ring0 + (uint32_t)(w * (D * kSlot))) + (uint32_t)(lane * 16);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const float4 v = load_shared(theirs + nt * 512u);
                sum[nt][0] += v.x;
                sum[nt][1] += v.y;
                sum[nt][2] += v.z;
                sum[nt][3] += v.w;
            }
        }
    };
    if (CLUSTER) {   // one sum per tile, where the CTA that stores it finds it
        for (int tl = warp; tl < my_cnt; tl += kWarps) {
            float sum[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[nt][i] = 0.0f;
            add_warps(sum, tl);
            put(smem0 + (uint32_t)(p.off_red + tl * (NT * 512)), sum);
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (rp > 0 && t0 < my_cnt) wait(tbar);
    const __half* ts = reinterpret_cast<const __half*>(smem + p.off_t);
#pragma unroll 1
    for (int tl = t0; tl < my_cnt; tl += t_step) {
        float sum[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[nt][i] = 0.0f;
        for (int j0 = 0; j0 < rp; j0 += 64) {
            if (tl != t0 || j0 > 0)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (j0 + q * 16 < rp) load_a(a0[q], tl, j0 + q * 16);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j0 + q * 16 < rp) {
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const __half* trow = ts + (nt * 8 + gq) * rp + j0 + q * 16 + 2 * tg;
                        mma_f16(sum[nt], a0[q], *reinterpret_cast<const uint32_t*>(trow), *reinterpret_cast<const uint32_t*>(trow + 8));
                    }
                }
        }
        if (!CLUSTER) add_warps(sum, tl);
        for (int r = 0; CLUSTER && r < C; ++r) {
            float4 v[NT];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) v[nt] = load_from_rank(smem0 + (uint32_t)(p.off_red + tl * (NT * 512) + (nt * 32 + lane) * 16), (uint32_t)r);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                sum[nt][0] += v[nt].x;
                sum[nt][1] += v[nt].y;
                sum[nt][2] += v[nt].z;
                sum[nt][3] += v[nt].w;
            }
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int tk = nt * 8 + 2 * tg + (i & 1);
                if (tk < p.T) {
                    const size_t o = (size_t)tk * p.ldy + (size_t)(my_start + tl) * 16 + gq + 8 * (i >> 1);
                    if (p.out_f32) reinterpret_cast<float*>(p.y)[o] = sum[nt][i];
                    else reinterpret_cast<__nv_bfloat16*>(p.y)[o] = __float2bfloat16_rn(sum[nt][i]);
                }
            }
    }
    // (no CTA leaves while another reads its sums)
    if (CLUSTER) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int BITS, int NT, int PER, int D, bool CLUSTER, typename SIBS>
__global__ void __launch_bounds__(kWarps * 32, 1)
run_kernel(const RunParams p_in, const __grid_constant__ SIBS sibs) {
    RunParams p = p_in;
    const int2 cta = select_sibling(p, CLUSTER ? (int)blockIdx.x / p.cluster : (int)blockIdx.x, sibs);
    // experts of a mixture layer: those with at most eight rows take one token tile although another of the launch needs two
    if (NT == 2 && !CLUSTER && sizeof(SIBS) > 1 && p.T <= 8) run_body<BITS, 1, PER, D, CLUSTER>(p, cta);
    else run_body<BITS, NT, PER, D, CLUSTER>(p, cta);
}

struct RunPlan {
    int nt, per, depth, units, cluster, most;   // units: clusters of the grid; most: row tiles of a cluster
    int off_t, off_red, off_x, x_bytes, off_ring, smem_bytes;
    int cta0[kMaxSiblings];
};

// The persistent CTAs are shared out in proportion to the layers' row tiles (at least one CTA each): the first CTA (cluster) of layers
// 1 .. n and, returned, the most tiles of one.  mixed: experts of up to eight rows run the loop of one token tile beside others that run
// that of two; a tile of the latter counts one and a half.  (Where every layer runs one loop this share left the smaller experts behind:
// 2048 -> 5632, 4 bits, eight experts of 20 and 4 rows 38.0 us and with even shares 33.8; 8192 -> 5632, 2 bits, 12 and 4 rows, two CTAs
// sharing K, 73.3 and 60.4.)
int share_ctas(const lopro_desc& d, const StreamSiblingArgs* more, int grid, bool mixed, int* cta0) {
    const int n = more != nullptr ? more->n : 0;
    auto tiles = [&](int i) { return (i == 0 ? d.d_out : more->d_out[i - 1]) / 16; };
    auto cost = [&](int i) { return (long long)tiles(i) * (mixed && more->T_of[i] <= 8 ? 2 : 3); };
    long long all = 0, before = 0;
    for (int i = 0; i <= n; ++i) all += cost(i);
    int most = 0, from = 0;
    for (int i = 0; i <= n; ++i) {
        int to = grid;
        before += cost(i);
        if (i < n) {
            to = (int)((before * grid + all / 2) / all);
            const int lo = from + 1, hi = grid - (n - i);
            if (to < lo) to = lo;
            if (to > hi) to = hi;
            cta0[i] = to;
        }
        const int here = (tiles(i) + to - from - 1) / (to - from);
        if (here > most) most = here;
        from = to;
    }
    return most;
}

bool plan_run(const lopro_desc& d, int T, const StreamSiblingArgs* more, RunPlan* pl) {
    if (T < 1 || T > kDecodeMaxT) return false;
    pl->nt = T <= 8 ? 1 : (T <= 16 ? 2 : 4);
    const int r_pad = d.rank > 0 ? round_up_int(d.rank, 16) : 0, ktok = pl->nt * 8, nsteps = d.d_in / 64;
    pl->x_bytes = T * kActRecord;   // (rows beyond the tokens are read, not used: the last stage has room behind it)
    const int forms[2][3][2] = {{{4, 3}, {4, 2}, {2, 3}}, {{2, 4}, {2, 3}, {2, 2}}};   // (steps of a batch, batches of a ring)
    for (int c = 1; c <= 2; c *= 2) {   // CTAs of a cluster: as few as it takes to hold the activations
        pl->cluster = c;
        pl->units = sm_count() / c;
        if (more != nullptr && more->n + 1 > pl->units) continue;
        pl->most = share_ctas(d, more, pl->units, more != nullptr && more->own_rows && pl->nt == 2 && c == 1, pl->cta0);
        for (const auto& f : forms[pl->nt == 4]) {
            pl->per = f[0];
            pl->depth = f[1];
            if (nsteps % pl->per != 0 || nsteps / pl->per < c) continue;
            if (pl->depth * pl->per * (128 * d.bits + 64) < pl->nt * 512) continue;   // a warp's last sums go where its ring was
            int stages = 0;   // of activations that a CTA's part of K touches, at most
            for (int r = 0; r < c; ++r) {
                const int nb = nsteps / pl->per, k0 = nb * r / c * pl->per, k1 = nb * (r + 1) / c * pl->per, n = (k1 + 15) / 16 - k0 / 16;
                if (n > stages) stages = n;
            }
            if (stages > kMaxX) continue;
            int off = 0;
            pl->off_t = off;
            off += round_up_int(ktok * r_pad * 2, 128);
            pl->off_red = off;
            off += pl->most * pl->nt * 512;
            pl->off_ring = off;
            off += round_up_int(kWarps * pl->depth * pl->per * (128 * d.bits + 64), 128);
            pl->off_x = off;
            off += stages * pl->x_bytes + (ktok - T) * kActRecord;
            pl->smem_bytes = off;
            if (off <= kRunMaxSmem) return true;
        }
    }
    return false;
}

template <int BITS, int NT, int PER, int D, bool CLUSTER, typename SIBS>
cudaError_t launch_run_ks(const RunParams& p, const SIBS& sibs, const RunPlan& pl, cudaStream_t s) {
    static unsigned long long attr_done = 0;
    const auto kernel = run_kernel<BITS, NT, PER, D, CLUSTER, SIBS>;
    cudaError_t e = ensure_dynamic_smem(kernel, kRunMaxSmem, &attr_done);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.units * pl.cluster);
    cfg.blockDim = dim3(kWarps * 32);
    cfg.dynamicSmemBytes = pl.smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = pl.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CLUSTER ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, p, sibs);
}

template <int BITS, int NT, int PER, int D, bool CLUSTER>
cudaError_t launch_run_c(const RunParams& p, const RunSiblings& sibs, const RunPlan& pl, cudaStream_t s) {
    return sibs.n == 0 ? launch_run_ks<BITS, NT, PER, D, CLUSTER, NoRunSiblings>(p, NoRunSiblings{}, pl, s)
                       : launch_run_ks<BITS, NT, PER, D, CLUSTER, RunSiblings>(p, sibs, pl, s);
}
template <int BITS, int NT, int PER, int D>
cudaError_t launch_run_k(const RunParams& p, const RunSiblings& sibs, const RunPlan& pl, cudaStream_t s) {
    return pl.cluster > 1 ? launch_run_c<BITS, NT, PER, D, true>(p, sibs, pl, s) : launch_run_c<BITS, NT, PER, D, false>(p, sibs, pl, s);
}

template <int BITS>
cudaError_t launch_run_bits(const RunParams& p, const RunSiblings& sibs, const RunPlan& pl, cudaStream_t s) {
    if (pl.nt == 1) {
        if (pl.per == 2) return launch_run_k<BITS, 1, 2, 3>(p, sibs, pl, s);
        return pl.depth == 3 ? launch_run_k<BITS, 1, 4, 3>(p, sibs, pl, s) : launch_run_k<BITS, 1, 4, 2>(p, sibs, pl, s);
    }
    if (pl.nt == 2) {
        if (pl.per == 2) return launch_run_k<BITS, 2, 2, 3>(p, sibs, pl, s);
        return pl.depth == 3 ? launch_run_k<BITS, 2, 4, 3>(p, sibs, pl, s) : launch_run_k<BITS, 2, 4, 2>(p, sibs, pl, s);
    }
    // (a ring has room for the sums of four token tiles)
    if (pl.depth == 4) return launch_run_k<BITS, 4, 2, 4>(p, sibs, pl, s);
    if constexpr (3 * slot_bytes<BITS, 2>() >= 2048)
        if (pl.depth == 3) return launch_run_k<BITS, 4, 2, 3>(p, sibs, pl, s);
    if constexpr (2 * slot_bytes<BITS, 2>() >= 2048)
        if (pl.depth == 2) return launch_run_k<BITS, 4, 2, 2>(p, sibs, pl, s);
    return cudaErrorInvalidValue;
}

}  // namespace

int warp_run_steps(const lopro_desc& d, int T, const StreamSiblingArgs* more, int32_t (&form)[5]) {
    RunPlan pl;
    if (option(LOPRO_OPT_NO_STEP_RUNS) == 1 || !plan_run(d, T, more, &pl)) return 0;
    form[0] = pl.nt;
    form[1] = pl.per;
    form[2] = pl.depth;
    form[3] = pl.cluster;
    form[4] = pl.most;
    return pl.most * (d.d_in / 64) / pl.cluster;
}

cudaError_t launch_warp_runs(const lopro_desc& d, const uint8_t* blob, const BlobLayout& L, const uint8_t* ws,
                        const WorkspaceLayout& W, void* y, int64_t ldy, int out_dtype, int T, cudaStream_t s, int t0,
                        const StreamSiblingArgs* more) {
    RunPlan pl;
    if (!plan_run(d, T, more, &pl)) return cudaErrorInvalidValue;
    RunParams p;
    p.codes = blob + L.off[LOPRO_SEC_CODES];
    p.sz = blob + L.off[LOPRO_SEC_SCALEZERO];
    p.A = blob + L.off[LOPRO_SEC_A];
    // t0: first token of this launch within the activation image and t (a chunk of a longer batch)
    p.act = ws + W.off_xrot + (size_t)t0 * kActRecord;
    p.t = reinterpret_cast<const __half*>(ws + W.off_t) + (size_t)t0 * (d.rank > 0 ? L.r_pad : 0);
    p.status = reinterpret_cast<int*>(const_cast<uint8_t*>(ws) + W.off_status);
    p.y = y;
    p.ldy = ldy;
    p.out_f32 = out_dtype == LOPRO_OUT_F32;
    p.m = d.d_out;
    p.T = T;
    p.t_pad = W.t_pad;
    p.nsteps = d.d_in / 64;
    int gs = d.group_size / 64, gshift = 0;
    while ((1 << gshift) < gs) ++gshift;
    p.gshift = gshift;
    p.r_pad = d.rank > 0 ? L.r_pad : 0;
    p.lr8 = d.lowrank_format == LOPRO_LOWRANK_FP8 ? 1 : 0;
    p.n_clusters = pl.units;
    p.cluster = pl.cluster;
    p.off_t = pl.off_t;
    p.off_red = pl.off_red;
    p.off_x = pl.off_x;
    p.x_bytes = pl.x_bytes;
    p.off_ring = pl.off_ring;
    RunSiblings sibs = {};
    if (more != nullptr && more->n > 0) {
        sibs.n = more->n;
        for (int i = 0; i < more->n; ++i) {
            sibs.cta0[i] = pl.cta0[i];
            const uint8_t* b = more->blob[i];
            const BlobLayout& Li = more->L[i];
            const uint8_t* wsi = more->ws[i];
            sibs.codes[i] = b + Li.off[LOPRO_SEC_CODES];
            sibs.sz[i] = b + Li.off[LOPRO_SEC_SCALEZERO];
            sibs.A[i] = b + Li.off[LOPRO_SEC_A];
            sibs.act[i] = wsi + W.off_xrot + (size_t)t0 * kActRecord;
            sibs.t[i] = reinterpret_cast<const __half*>(wsi + W.off_t) + (size_t)t0 * (d.rank > 0 ? L.r_pad : 0);
            sibs.y[i] = more->y[i];
            sibs.ldy[i] = more->ldy[i];
            sibs.m[i] = more->d_out[i];
            sibs.T[i] = more->own_rows ? more->T_of[i + 1] : T;
        }
    }
    if (more != nullptr && more->own_rows) p.T = more->T_of[0];  // also where this expert is the only one of its launch
    switch (d.bits) {
        case 2: return launch_run_bits<2>(p, sibs, pl, s);
        case 3: return launch_run_bits<3>(p, sibs, pl, s);
        default: return launch_run_bits<4>(p, sibs, pl, s);
    }
}

}  // namespace lopro
