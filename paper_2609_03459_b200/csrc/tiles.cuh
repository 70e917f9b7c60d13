// 64 x 64 output tiles of 3xTF32 products for shapes without a kernel of their own: staging of ragged rows with cp.async and
// the product of a warp's 32 x 32 quarter.  Pitches of 72 (fragments run down the rows) and 36 floats (along the rows) keep
// the fragment loads free of bank conflicts; every k step is added in rounded fp32 (tt_mma_3xtf32_rounded).
#pragma once
#include "common.cuh"
#include "mma.cuh"

#define MT_EDGE 64
#define MT_KROWS 32
#define MT_PA (MT_EDGE + 8)
#define MT_PC (MT_KROWS + 4)

// 4-byte asynchronous copy global -> shared
__device__ __forceinline__ void tt_cp_async4(void* smem_dst, const void* gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gsrc) : "memory");
}

// dst[row][0 .. 4 * W4) = src[row][off .. off + avail), the rest of the row (and rows without a source) zero; 128 threads
template <int ROWS, int W4>
__device__ __forceinline__ void tt_stage_rows(float* dst, int pitch, const float* const* src, int off, int avail, bool vec)
{
    if (vec) {
        for (int i = threadIdx.x; i < ROWS * W4; i += 128) {
            const int row = i / W4, c4 = i % W4;
            const float* p = src[row];
            float* d = dst + row * pitch + 4 * c4;
            if (p && 4 * c4 < avail) tt_cp_async16(d, p + off + 4 * c4);
            else *reinterpret_cast<float4*>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
        for (int i = threadIdx.x; i < ROWS * W4 * 4; i += 128) {
            const int row = i / (W4 * 4), c = i % (W4 * 4);
            const float* p = src[row];
            float* d = dst + row * pitch + c;
            if (p && c < avail) tt_cp_async4(d, p + off + c);
            else *d = 0.f;
        }
    }
}

// sum += A . B over 8 k values: mtl row tiles of 16, ntl column blocks of 8.  The A fragment of row tile mt is
// {a0, a1, a2, a3}[16 mt * astep], the B fragment of block nt {b0, b1}[8 nt * bstep].  WHOLE: for shapes that fill their tiles; then four
// products at a time, whose chains of three instructions overlap (with a branch around each tile the compiler left them one after the
// other: rank 64, four cores, 65 k lookups, the two middle levels 133.7 to 128.4 us; one kernel with both ways would cost
// shapes of partial tiles 6 us of 52: 3x3x5, ranks 6 and 4, 1 M lookups)
template <bool WHOLE>
__device__ __forceinline__ void tt_quarter_step(float (&sum)[2][4][4], const float* a0, const float* a1, const float* a2, const float* a3,
                                                int astep, const float* b0, const float* b1, int bstep, int mtl, int ntl)
{
    Tf32Pair a[2][4];
    if (WHOLE && mtl == 2 && ntl == 4) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            a[mt][0] = tt_split_tf32(a0[16 * mt * astep]);
            a[mt][1] = tt_split_tf32(a1[16 * mt * astep]);
            a[mt][2] = tt_split_tf32(a2[16 * mt * astep]);
            a[mt][3] = tt_split_tf32(a3[16 * mt * astep]);
        }
#pragma unroll
        for (int np = 0; np < 4; np += 2) {
            Tf32Pair b[2][2];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                b[nt][0] = tt_split_tf32(b0[8 * (np + nt) * bstep]);
                b[nt][1] = tt_split_tf32(b1[8 * (np + nt) * bstep]);
            }
            float d[2][2][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) tt_mma_tf32_zero(d[mt][nt], a[mt][0].lo, a[mt][1].lo, a[mt][2].lo, a[mt][3].lo, b[nt][0].hi, b[nt][1].hi);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) tt_mma_tf32(d[mt][nt], a[mt][0].hi, a[mt][1].hi, a[mt][2].hi, a[mt][3].hi, b[nt][0].lo, b[nt][1].lo);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) tt_mma_tf32(d[mt][nt], a[mt][0].hi, a[mt][1].hi, a[mt][2].hi, a[mt][3].hi, b[nt][0].hi, b[nt][1].hi);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) sum[mt][np + nt][i] += d[mt][nt][i];
        }
        return;
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
        if (mt < mtl) {
            a[mt][0] = tt_split_tf32(a0[16 * mt * astep]);
            a[mt][1] = tt_split_tf32(a1[16 * mt * astep]);
            a[mt][2] = tt_split_tf32(a2[16 * mt * astep]);
            a[mt][3] = tt_split_tf32(a3[16 * mt * astep]);
        }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
        if (nt < ntl) {
            Tf32Pair b[2];
            b[0] = tt_split_tf32(b0[8 * nt * bstep]);
            b[1] = tt_split_tf32(b1[8 * nt * bstep]);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
                if (mt < mtl) tt_mma_3xtf32_rounded(sum[mt][nt], a[mt], b);
        }
}

