// The register tile of the CUDA-core fp32 contractions.  A block's operand tiles sit in
// shared memory k by k: A as pairs (a, a), B plain, so that one packed FMA
// (fma.rn.f32x2: two IEEE fp32 FMAs in one instruction) takes a pair of columns without any
// register shuffling.  Every sum is the fp32 FMA chain over ascending k.
//
// A thread holds TM rows x TN columns (multiples of 4), in groups of four rows RS apart and
// four columns CS apart: a quarter warp then reads 16-byte pieces of neighbouring columns (no
// bank conflicts) and broadcasts its rows.  At 8 x 8 a k costs 6 shared-memory loads for
// 32 packed FMAs (scalar FMAs: 4 loads for 64).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mure {

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}

__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// acc[i][j]: row i, columns (2j, 2j + 1) of the thread.  a: the tile's first k line at the
// thread's first row, BM pairs per k; b: the same for its first column, BN floats per k.
template <int KN, int BM, int BN, int TM, int TN, int RS, int CS>
__device__ __forceinline__ void simt_tile_fma(f32x2 (&acc)[TM][TN / 2], const float2 *a, const float *b)
{
#pragma unroll 2
    for (int k = 0; k < KN; ++k) {
        f32x2 av[TM], bv[TN / 2];
#pragma unroll
        for (int i = 0; i < TM; i += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(a + k * BM + (i / 4) * RS + (i & 3));
            av[i] = v.x;
            av[i + 1] = v.y;
        }
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(b + k * BN + (j / 4) * CS);
            bv[j / 2] = v.x;
            bv[j / 2 + 1] = v.y;
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) acc[i][j] = fma2(av[i], bv[j], acc[i][j]);
    }
}

}  // namespace mure
