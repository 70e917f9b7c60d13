// Intermediate products (paper Sec. 3.2, "Intermediate Computation") of several prefix groups at once on the
// tensor cores.
//
// Groups are walked in digit-major order, so neighbours share the slice B = G_{K-1}[i_{K-1}] (r_a x cols).  With
// P_{K-2} of MROWS = 4 (or 2) rows per group, NG = 16 / MROWS = 4 (or 8) groups stack into one 16 x r_a operand, and
//     [C_0; ..; C_{NG-1}] = [P_0; ..; P_{NG-1}] . B
// is a 16 x cols product of m16n8k8 tiles in 3xTF32 (see mma.cuh).  The slice then enters the SM once per NG
// groups instead of once per group (the FP32-pipe form of this product was bound by the L1 operand path), and the
// product leaves the FP32 pipe.  Groups of the batch that use another slice (a run boundary) are handled in a
// further pass; rows of groups that are not part of a pass are zero and their result is not stored.
#pragma once
#include "mma.cuh"

// `hook` runs once per batch after its first block of columns: loads that the caller has under way by then are waited for
// under the products of the other blocks.
struct QuadNothing { __device__ __forceinline__ void operator()() const {} };

// One pass.  Lane (g = lane / 4, t = lane % 4) feeds rows g and g + 8 of the stacked operand: row g belongs to group
// g / MROWS (source srcA, taken when selA), row g + 8 to group (8 + g) / MROWS (srcB, selB); m = g % MROWS is the row
// of P inside the group.  src points at P (MROWS x ra, row-major).  ra <= 8 * KTMAX, any value (the k range is padded
// with zeros).  Results go to the group's C tile in Cs4, stored as [PM][RB + 4]: rows of r_{K-1} = RB values padded by four
// floats, which makes the row stage's fragment loads from shared memory conflict-free.
//
// Column mapping: a block of 32 columns is one float4 load per lane and k row (8 lanes x 16 bytes = 128 bytes per
// row); tile j of the block takes component j, i.e. tile column n' stands for slice column 32 * block + 4 n' + j, so
// that a lane ends up with 8 consecutive columns of each of its two rows (two float4 stores per row).
template <int COLS, int MROWS, int KTMAX, int RB, class Hook>
__device__ __forceinline__ void tt_quad_mid_mma(const float* __restrict__ B, int ra, const float* __restrict__ srcA,
                                                const float* __restrict__ srcB, bool selA, bool selB, float* Cs4, int lane, Hook& hook)
{
    static_assert((MROWS == 2 || MROWS == 4) && KTMAX % 2 == 0, "stacking of 8 or 4 groups");
    const int g = lane >> 2, t = lane & 3, m = g & (MROWS - 1);
    const int kta = (ra + 7) >> 3;
    // the stacked operand stays unsplit in registers (KTMAX * 4) and is split where it is used: half the registers of
    // pre-split fragments, which buys a resident CTA more per SM
    float araw[KTMAX][4];
#pragma unroll
    for (int kt = 0; kt < KTMAX; ++kt) {
        const int k0 = 8 * kt + t, k1 = k0 + 4;
        araw[kt][0] = (selA && k0 < ra) ? __ldg(srcA + m * ra + k0) : 0.f;
        araw[kt][1] = (selB && k0 < ra) ? __ldg(srcB + m * ra + k0) : 0.f;
        araw[kt][2] = (selA && k1 < ra) ? __ldg(srcA + m * ra + k1) : 0.f;
        araw[kt][3] = (selB && k1 < ra) ? __ldg(srcB + m * ra + k1) : 0.f;
    }
    const float4* __restrict__ B4 = reinterpret_cast<const float4*>(B);
    constexpr int C4N = COLS / 4;
    constexpr int DSUB = COLS / RB;                             // d_{K-1}: rows of C per row of P
    constexpr int TILE = MROWS * DSUB * (RB + 4);
    float* dstA = Cs4 + (size_t)(g / MROWS) * TILE;
    float* dstB = Cs4 + (size_t)((8 + g) / MROWS) * TILE;
    // offset of columns [32 nb + 8 t, + 8) of row m inside a tile
    auto coff = [&](int nb) {
        const int col = 32 * nb + 8 * t;
        return (m * DSUB + col / RB) * (RB + 4) + col % RB;
    };
#pragma unroll 1
    for (int nb = 0; nb < COLS / 32; ++nb) {
        float acc[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[j][0] = 0.f; acc[j][1] = 0.f; acc[j][2] = 0.f; acc[j][3] = 0.f; }
#pragma unroll
        for (int kc = 0; kc < KTMAX; kc += 2) {   // two k steps (16 rows of B) in flight at a time
            float4 f[2][2];
#pragma unroll
            for (int kt = 0; kt < 2; ++kt) {
                const int k0 = 8 * (kc + kt) + t, k1 = k0 + 4;
                f[kt][0] = k0 < ra ? __ldg(B4 + (size_t)k0 * C4N + 8 * nb + g) : make_float4(0.f, 0.f, 0.f, 0.f);
                f[kt][1] = k1 < ra ? __ldg(B4 + (size_t)k1 * C4N + 8 * nb + g) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int kt = 0; kt < 2; ++kt) {
                if (kc + kt < kta) {
                    Tf32Pair a[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) a[x] = tt_split_tf32(araw[kc + kt][x]);
                    const float v0[4] = {f[kt][0].x, f[kt][0].y, f[kt][0].z, f[kt][0].w};
                    const float v1[4] = {f[kt][1].x, f[kt][1].y, f[kt][1].z, f[kt][1].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        Tf32Pair b[2];
                        b[0] = tt_split_tf32(v0[j]);
                        b[1] = tt_split_tf32(v1[j]);
                        tt_mma_3xtf32(acc[j], a, b);
                    }
                }
            }
        }
        if (nb == 0) hook();
        if (selA) {
            *reinterpret_cast<float4*>(dstA + coff(nb)) = make_float4(acc[0][0], acc[1][0], acc[2][0], acc[3][0]);
            *reinterpret_cast<float4*>(dstA + coff(nb) + 4) = make_float4(acc[0][1], acc[1][1], acc[2][1], acc[3][1]);
        }
        if (selB) {
            *reinterpret_cast<float4*>(dstB + coff(nb)) = make_float4(acc[0][2], acc[1][2], acc[2][2], acc[3][2]);
            *reinterpret_cast<float4*>(dstB + coff(nb) + 4) = make_float4(acc[0][3], acc[1][3], acc[2][3], acc[3][3]);
        }
    }
}

// All passes of one batch of cnt <= 16 / MROWS groups.  Lane q < cnt holds group q's slice index (imq) and operand
// pointer (srcq).
template <int COLS, int MROWS, int KTMAX, int RB, class Hook = QuadNothing>
__device__ __forceinline__ void tt_quad_mid(const float* __restrict__ core_mid, size_t slice_floats, int ra, int cnt, uint32_t imq,
                                            const float* srcq, float* Cs4, int lane, Hook hook = Hook())
{
    bool pending = true;
    auto once = [&]() { if (pending) hook(); pending = false; };
    const int g = lane >> 2;
    const int qA = g / MROWS, qB = (8 + g) / MROWS;
    const unsigned long long sp = (unsigned long long)reinterpret_cast<uintptr_t>(srcq);
    const float* srcA = reinterpret_cast<const float*>((uintptr_t)__shfl_sync(0xffffffffu, sp, qA));
    const float* srcB = reinterpret_cast<const float*>((uintptr_t)__shfl_sync(0xffffffffu, sp, qB));
    unsigned remaining = (1u << cnt) - 1u;
    while (remaining) {
        const int first = __ffs(remaining) - 1;
        const uint32_t im = __shfl_sync(0xffffffffu, imq, first);
        const unsigned sel = __ballot_sync(0xffffffffu, lane < 16 / MROWS && ((remaining >> lane) & 1u) && imq == im) & ((1u << (16 / MROWS)) - 1u);
        const bool selA = (sel >> qA) & 1u, selB = (sel >> qB) & 1u;
        tt_quad_mid_mma<COLS, MROWS, KTMAX, RB>(core_mid + (size_t)im * slice_floats, ra, srcA, srcB, selA, selB, Cs4, lane, once);
        remaining &= ~sel;
    }
}

// The same in fp32 for slices of 32 columns (rank 8, C of 16 rows), of up to four groups with any slices: eight lanes per group, each
// with four columns of its four rows.  The backward rebuilds C from these: its sums are those that it had before the products of
// neighbouring groups were formed together, four terms apart, then pairwise.
template <int RB, class Hook>
__device__ __forceinline__ void tt_quad_mid_fp32(const float* __restrict__ core_mid, size_t slice_floats, int ra, int cnt, uint32_t imq,
                                                 const float* srcq, float* Cs4, int lane, Hook hook)
{
    static_assert(RB == 8, "a group's 32 columns are eight float4s");
    const int q = lane >> 3, c4 = lane & 7;
    const bool on = q < cnt;
    const uint32_t im = __shfl_sync(0xffffffffu, imq, q);
    const float* src = reinterpret_cast<const float*>((uintptr_t)__shfl_sync(0xffffffffu, (unsigned long long)reinterpret_cast<uintptr_t>(srcq), q));
    const float4* __restrict__ B4 = reinterpret_cast<const float4*>(core_mid + (size_t)im * slice_floats) + c4;
    float4 acc[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int a0 = 0; a0 < ra; a0 += 8) {
        float4 b[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) b[a] = on && a0 + a < ra ? __ldg(B4 + (size_t)(a0 + a) * 8) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (a0 == 0) hook();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            float x[8];
            const float* __restrict__ row = src + m * ra + a0;
            if ((ra & 3) == 0) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 v = on && a0 + 4 * h < ra ? __ldg(reinterpret_cast<const float4*>(row) + h) : make_float4(0.f, 0.f, 0.f, 0.f);
                    x[4 * h] = v.x; x[4 * h + 1] = v.y; x[4 * h + 2] = v.z; x[4 * h + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int a = 0; a < 8; ++a) x[a] = on && a0 + a < ra ? __ldg(row + a) : 0.f;
            }
            auto sum = [&](float b0, float b1, float b2, float b3, float b4, float b5, float b6, float b7) {
                return (fmaf(x[4], b4, x[0] * b0) + fmaf(x[5], b5, x[1] * b1)) + (fmaf(x[6], b6, x[2] * b2) + fmaf(x[7], b7, x[3] * b3));
            };
            acc[m].x += sum(b[0].x, b[1].x, b[2].x, b[3].x, b[4].x, b[5].x, b[6].x, b[7].x);
            acc[m].y += sum(b[0].y, b[1].y, b[2].y, b[3].y, b[4].y, b[5].y, b[6].y, b[7].y);
            acc[m].z += sum(b[0].z, b[1].z, b[2].z, b[3].z, b[4].z, b[5].z, b[6].z, b[7].z);
            acc[m].w += sum(b[0].w, b[1].w, b[2].w, b[3].w, b[4].w, b[5].w, b[6].w, b[7].w);
        }
    }
    if (on) {
        float* dst = Cs4 + (size_t)q * (16 * (RB + 4)) + (c4 >> 1) * (RB + 4) + 4 * (c4 & 1);   // columns 4 c4 .. of row m: row 4 m + c4 / 2 of C
#pragma unroll
        for (int m = 0; m < 4; ++m) *reinterpret_cast<float4*>(dst + (size_t)m * (4 * (RB + 4))) = acc[m];
    }
}
