// The rank-1 randomized sketch (sketch.cu) as seen by the offline side's entry points (quantize.cu).
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace lopro {

struct SketchJob {
    const float* w;          // [m][n] matrix to decompose, read only
    const float* sketches;   // [r][n]
    const float* s;          // scale of the columns (null: ones)
    float* s_eff;            // [n] the scale as applied, or null
    __half* s16;             // [n] the scale rounded to fp16 (then applied in that form), or null
    float *U, *sigma, *V;    // outputs [m][r], [r], [r][n]; V 16-byte aligned
    int* status;             // LOPRO_ERR_TIMEOUT where a wait ran out (the launch clears the scratch's own word only)
    int m, n, r, it, cast;
};

bool sketch_supported(int n, int r);
size_t sketch_scratch_bytes(int m, int n, int r);
inline int* sketch_status(void* scratch) { return (int*)scratch; }  // a status word that the launch clears
cudaError_t launch_sketch(const SketchJob& job, void* scratch, cudaStream_t s);
// w <- w - U diag(sigma) V, unless *status is an error
cudaError_t launch_deflate(float* w, int m, int n, int r, const float* U, const float* sigma, const float* V, const int* status,
                           cudaStream_t s);

// fp32 -> nearest fp8 e4m3 value (ties to even, saturating), returned as fp32; bits optionally kept.
__device__ __forceinline__ float round_e4m3(float x, unsigned char* bits = nullptr) {
    unsigned short pair;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(pair) : "f"(0.0f), "f"(x));  // low byte = second operand
    if (bits) *bits = (unsigned char)(pair & 0xffu);
    const uint32_t h2 = e4m3x2_to_f16x2((unsigned short)(pair & 0xffu));
    return __half2float(__ushort_as_half((unsigned short)(h2 & 0xffffu)));
}

}  // namespace lopro
