// Forward path: prefix products, fused last-two-level contraction, bag pooling.
//
// Work is organised around the sorted prefix tree built by the grouping pass.  A "group" is a node of
// level K-1 (a distinct (i_1..i_{K-1}) prefix); its children are the distinct rows that share it.
//   * schedule (grouping.cu, group_cluster.cu): cost(group) = c_mid + children * c_last (FMA counts), exclusive scan, and
//     every table is cut into `units` slices of equal cost (or equal counts); one CTA per unit, dispatched dynamically by
//     the hardware.
//   * contraction: per group the partial product C = P_{K-2} . G_{K-1}[i_{K-1}] is formed once in shared
//     memory (paper Sec. 3.2 "Intermediate Computation") and every child row E = C . G_K[i_K] is produced
//     from it ("Embedding Computation"); C never goes to global memory.
//   * pooling ("Vector Aggregation"): one warp per bag gathers its rows through the rank structure and
//     reduces them in registers; lanes of different sub-warps are combined with warp shuffles.  No atomics.
#include "common.cuh"
#include "scan.cuh"
#include "mma.cuh"
#include "quad_mid.cuh"
#include "generic.cuh"
#include "wide.cuh"
#include "tiles.cuh"

// ---------------------------------------------------------------------------------------------- products

// P_2 for every level-2 node of a four-core table: P_2 = G_1[i_1] . G_2[i_2].  A CTA keeps to one i_2 and 64 columns of its
// slice, looks for the present i_1 in the level's bitmap, LEVEL2_SCAN of them at a time (a prefix's node is a rank look-up
// there, so the nodes of one i_2 need no list), and multiplies the slices that it found, 64 stacked rows at a time
// with fp32 FMAs: a thread makes eight rows by four columns, in the order of tt_mid_product (3xTF32 tiles took the same time, the
// staging bounds both, and put the error of `out` against 64 bits at 1.29e-7 instead of 1.09e-7 for 3x3x3x5, rank 9).  One CTA
// per node reads its slice for itself: 3403 nodes of 2 x 64 by 64 x 256 took 70 us, bound by 0.2 GB of slices from L2, and
// take 16 us this way.
#define LEVEL2_SCAN 256
// CTAs that share the first digits of one i_2, a block of LEVEL2_SCAN each in turn (popular prefixes are often the first ones)
__host__ __device__ __forceinline__ uint32_t tt_level2_parts(const TableDesc& td)
{
    const uint32_t most = ((uint32_t)td.n[0] + LEVEL2_SCAN - 1) / LEVEL2_SCAN, want = 2048u / (uint32_t)td.n[1];
    return want < 1u ? 1u : (want < most ? want : most);
}
__global__ void __launch_bounds__(128, 4) k_level2(WsView w)
{
    tt_pdl_enter();
    __shared__ __align__(16) float sm[2 * (MT_EDGE * MT_PC + MT_KROWS * MT_PA)];
    __shared__ const float* s_row[MT_EDGE];     // rows of G_1
    __shared__ float* s_out[MT_EDGE];
    __shared__ const float* s_slice[128];       // rows of the slice of G_2
    __shared__ uint2 s_list[LEVEL2_SCAN];       // present first digits and their nodes
    __shared__ int s_count;
    const TableDesc& td = w.tdesc[blockIdx.y];
    const int M = td.d[0], ra = td.r[1], cols = td.d[1] * td.r[2], c0 = (int)blockIdx.z * MT_EDGE;
    const uint32_t n2 = (uint32_t)td.n[1], i2 = blockIdx.x % n2, part = blockIdx.x / n2, parts = tt_level2_parts(td);
    if (part >= parts || c0 >= cols) return;
    const uint32_t n1 = (uint32_t)td.n[0];
    const bool vec = (ra & 3) == 0 && (cols & 3) == 0;
    const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 4, tx = tid & 15;
    s_slice[tid] = tid < ra ? td.core[1] + (size_t)i2 * td.slice_floats[1] + (size_t)tid * cols + c0 : nullptr;   // r <= 128
    const int kpasses = (ra + MT_KROWS - 1) / MT_KROWS;
    const uint32_t count = w.counters[CTR_LEVEL0 + 2];
    constexpr int STAGE = MT_EDGE * MT_PC + MT_KROWS * MT_PA;
    for (uint32_t base = part * LEVEL2_SCAN; base < n1; base += parts * LEVEL2_SCAN) {
        if (tid == 0) s_count = 0;
        __syncthreads();
        uint2 e[LEVEL2_SCAN / 128];
#pragma unroll
        for (int j = 0; j < LEVEL2_SCAN / 128; ++j) {
            const uint32_t p = base + 128 * j + tid;
            e[j] = p < n1 ? w.bml[2][td.lword_base[2] + ((p * n2 + i2) >> 5)] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int j = 0; j < LEVEL2_SCAN / 128; ++j) {
            const uint32_t p = base + 128 * j + tid, bit = (p * n2 + i2) & 31;
            const uint32_t v = e[j].y + __popc(e[j].x & ((1u << bit) - 1u));
            const bool present = ((e[j].x >> bit) & 1u) && v < count;
            const unsigned found = __ballot_sync(0xffffffffu, present);
            int at = 0;
            if (lane == 0 && found) at = atomicAdd(&s_count, __popc(found));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (present) s_list[at + __popc(found & ((1u << lane) - 1u))] = make_uint2(p, v);
        }
        __syncthreads();
        const int rows = s_count * M;               // at most 256 x 1024
        for (int row0 = 0; row0 < rows; row0 += MT_EDGE) {
            if (tid < MT_EDGE) {
                const int q = (row0 + tid) / M, m = row0 + tid - q * M;
                const bool some = row0 + tid < rows;
                const uint2 x = some ? s_list[q] : make_uint2(0u, 0u);
                s_row[tid] = some ? td.core[0] + ((size_t)x.x * M + m) * ra : nullptr;
                s_out[tid] = some ? w.pbuf[2] + (size_t)x.y * w.stride[2] + (size_t)m * cols + c0 : nullptr;
            }
            __syncthreads();
            float sum[8][4];                        // rows ty + 8 i, columns 4 tx ..
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) sum[i][j] = 0.f;
            auto issue = [&](int kp) {
                float* st = sm + (kp & 1) * STAGE;
                tt_stage_rows<MT_EDGE, MT_KROWS / 4>(st, MT_PC, s_row, kp * MT_KROWS, ra - kp * MT_KROWS, vec);
                tt_stage_rows<MT_KROWS, MT_EDGE / 4>(st + MT_EDGE * MT_PC, MT_PA, s_slice + kp * MT_KROWS, 0, cols - c0, vec);
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            issue(0);
            for (int kp = 0; kp < kpasses; ++kp) {
                if (kp + 1 < kpasses) {
                    issue(kp + 1);
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                } else {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                }
                __syncthreads();
                const float* A = sm + (kp & 1) * STAGE + ty * MT_PC;
                const float* B = sm + (kp & 1) * STAGE + MT_EDGE * MT_PC + 4 * tx;
                const int kn = min(MT_KROWS, ra - kp * MT_KROWS);   // zeros up to the next multiple of four
                if (c0 + 4 * tx < cols)
#pragma unroll 2
                    for (int k = 0; k < kn; k += 4) {
                        float4 x[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const float4*>(A + 8 * i * MT_PC + k);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float4 y = *reinterpret_cast<const float4*>(B + (k + q) * MT_PA);
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const float f = q == 0 ? x[i].x : q == 1 ? x[i].y : q == 2 ? x[i].z : x[i].w;
                                sum[i][0] = fmaf(f, y.x, sum[i][0]); sum[i][1] = fmaf(f, y.y, sum[i][1]);
                                sum[i][2] = fmaf(f, y.z, sum[i][2]); sum[i][3] = fmaf(f, y.w, sum[i][3]);
                            }
                        }
                    }
                __syncthreads();
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float* out = s_out[ty + 8 * i];
                if (!out || c0 + 4 * tx >= cols) continue;
                out += 4 * tx;
                if ((cols & 3) == 0) *reinterpret_cast<float4*>(out) = make_float4(sum[i][0], sum[i][1], sum[i][2], sum[i][3]);
                else
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (c0 + 4 * tx + j < cols) out[j] = sum[i][j];
            }
            __syncthreads();   // the addresses are rewritten for the next tile
        }
        __syncthreads();   // all have read the count
    }
}

// Few nodes per slice, or few of the possible prefixes present; also the study switches, whose nodes no bitmap finds (every
// lookup or row its own).  One CTA per node
__global__ void __launch_bounds__(128) k_level2_nodes(WsView w)
{
    tt_pdl_enter();
    extern __shared__ float sm[];
    const uint32_t count = w.counters[CTR_LEVEL0 + 2];
    for (uint32_t v = blockIdx.x; v < count; v += gridDim.x) {
        const TableDesc& td = w.tdesc[tt_find_table(w.tb[2], w.T, v)];
        const int M = td.P[1], ra = td.r[1], cols = td.d[1] * td.r[2];
        const float* src = tt_left_operand(w, td, 2, v);
        for (int i = threadIdx.x; i < M * ra; i += blockDim.x) sm[i] = src[i];
        __syncthreads();
        const uint32_t ik = w.val[2][v] % (uint32_t)td.n[1];
        tt_mid_product(sm, td.core[1] + (size_t)ik * td.slice_floats[1], w.pbuf[2] + (size_t)v * w.stride[2], M, ra, cols);
        __syncthreads();
    }
}

// ---- register-tiled warp-level products (fast path) ---------------------------------------------------------
//
// One warp owns one group at a time.  FP32 FMA throughput is only reachable when every float that enters
// a lane's registers feeds >= 4 FMAs (the shared-memory / L1 path delivers 32 floats per clock per SM, the
// FMA pipes retire 128 lane-FMAs per clock), so:
//   * mid product  C = Pl . B : a lane owns 4 (or 8) consecutive columns of B for all M rows of Pl; B streams
//     through once as float4, Pl comes as float4 broadcasts from shared memory.
//   * last product E = C . D  : a lane keeps TP rows of C (TP x RB floats) in registers for the whole group
//     and streams the float4 rows of each child's D slice: 4*TP FMAs per loaded float4; PM/TP lanes cover a
//     row, so a warp produces 32*TP/PM rows at a time and each lane stores 4*TP consecutive floats of E.

// Cs[m*cols + c] = sum_a Pl[m][a] * Bsl[a*cols + c];  As holds Pl transposed: As[a*M + m].
// cols/4 must be a power of two and cols <= 128*CPL.
template <int M, int CPL>
__device__ __forceinline__ void tt_warp_mid(const float* As, const float* __restrict__ Bsl, float* Cs, int ra, int cols, int lane)
{
    const int c4n = cols >> 2;
    const int LA = (c4n / CPL) < 32 ? (c4n / CPL) : 32;  // lanes that cover one row of B
    const int NS = 32 / LA;                              // the a-range is split over NS lane groups
    const int s = lane / LA, ll = lane - s * LA;
    float acc[CPL][M][4];
#pragma unroll
    for (int i = 0; i < CPL; ++i)
#pragma unroll
        for (int m = 0; m < M; ++m) { acc[i][m][0] = 0.f; acc[i][m][1] = 0.f; acc[i][m][2] = 0.f; acc[i][m][3] = 0.f; }
    const float4* __restrict__ B4 = reinterpret_cast<const float4*>(Bsl);
#pragma unroll 16
    for (int a = s; a < ra; a += NS) {
        float4 b[CPL];
#pragma unroll
        for (int i = 0; i < CPL; ++i) b[i] = __ldg(B4 + (size_t)a * c4n + ll + i * LA);
        float av[M];
        if constexpr (M % 4 == 0) {
#pragma unroll
            for (int m4 = 0; m4 < M / 4; ++m4) {
                const float4 t = *reinterpret_cast<const float4*>(As + a * M + 4 * m4);
                av[4 * m4] = t.x; av[4 * m4 + 1] = t.y; av[4 * m4 + 2] = t.z; av[4 * m4 + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int m = 0; m < M; ++m) av[m] = As[a * M + m];
        }
#pragma unroll
        for (int i = 0; i < CPL; ++i)
#pragma unroll
            for (int m = 0; m < M; ++m) {
                acc[i][m][0] = fmaf(av[m], b[i].x, acc[i][m][0]);
                acc[i][m][1] = fmaf(av[m], b[i].y, acc[i][m][1]);
                acc[i][m][2] = fmaf(av[m], b[i].z, acc[i][m][2]);
                acc[i][m][3] = fmaf(av[m], b[i].w, acc[i][m][3]);
            }
    }
    for (int o = LA; o < 32; o <<= 1)
#pragma unroll
        for (int i = 0; i < CPL; ++i)
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[i][m][x] += __shfl_xor_sync(0xffffffffu, acc[i][m][x], o);
    if (s == 0) {
#pragma unroll
        for (int i = 0; i < CPL; ++i)
#pragma unroll
            for (int m = 0; m < M; ++m)
                *reinterpret_cast<float4*>(Cs + m * cols + 4 * (ll + i * LA)) = make_float4(acc[i][m][0], acc[i][m][1], acc[i][m][2], acc[i][m][3]);
    }
}

// E rows u0..u1 of the group whose C (PM x RB, row-major) is in Cs.  d_K = 4.
template <int PM, int RB, int TP>
__device__ __forceinline__ void tt_warp_rows(const float* Cs, const WsView& w, const TableDesc& td, uint32_t u0, uint32_t u1,
                                             uint32_t row_base, int lane)
{
    constexpr int LR = PM / TP;   // lanes per row
    constexpr int RW = 32 / LR;   // rows per batch
    const int q = lane % LR, slot = lane / LR;
    float c[TP][RB];
#pragma unroll
    for (int i = 0; i < TP; ++i)
#pragma unroll
        for (int b4 = 0; b4 < RB / 4; ++b4) {
            const float4 t = *reinterpret_cast<const float4*>(Cs + (TP * q + i) * RB + 4 * b4);
            c[i][4 * b4] = t.x; c[i][4 * b4 + 1] = t.y; c[i][4 * b4 + 2] = t.z; c[i][4 * b4 + 3] = t.w;
        }
    const int K = w.K;
    const float* __restrict__ GK = td.core[K - 1];
    const uint32_t* __restrict__ rows = w.val[K];
    for (uint32_t ub = u0; ub < u1; ub += RW) {
        const uint32_t u = ub + slot;
        const bool act = u < u1;
        const uint32_t iK = act ? rows[u] - row_base : 0u;
        const float4* __restrict__ D4 = reinterpret_cast<const float4*>(GK + (size_t)iK * (RB * 4));
        float acc[TP][4];
#pragma unroll
        for (int i = 0; i < TP; ++i) { acc[i][0] = 0.f; acc[i][1] = 0.f; acc[i][2] = 0.f; acc[i][3] = 0.f; }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const float4 d = __ldg(D4 + b);
#pragma unroll
            for (int i = 0; i < TP; ++i) {
                acc[i][0] = fmaf(c[i][b], d.x, acc[i][0]);
                acc[i][1] = fmaf(c[i][b], d.y, acc[i][1]);
                acc[i][2] = fmaf(c[i][b], d.z, acc[i][2]);
                acc[i][3] = fmaf(c[i][b], d.w, acc[i][3]);
            }
        }
        if (act) {
            float4* e = reinterpret_cast<float4*>(w.E + (size_t)u * (PM * 4) + TP * q * 4);
#pragma unroll
            for (int i = 0; i < TP; ++i) e[i] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        }
    }
}

// Tensor-core form of the last product (d_K = 4): E_u[p][j] = sum_b C[p][b] * D_u[b][j] as m16n8k8 tiles with
// M = 16 rows p of C, K = 8 values of b, N = 8 = two child rows x 4 columns j.  The fragments of C (split into TF32
// head and tail) stay in PM*RB/8 registers for the whole group; each child's slice is read exactly once per warp
// (two coalesced 64-byte pieces per load instruction), so the shared-memory / L1 path carries 4x fewer bytes per
// FMA than the FP32-pipe form and a warp needs ~1/3 of its registers.
template <int PM, int RB, int CS = RB>   // CS: row stride of C in shared memory
__device__ __forceinline__ void tt_warp_rows_mma(const float* Cs, const WsView& w, const TableDesc& td, uint32_t u0, uint32_t u1,
                                                 uint32_t row_base, int lane)
{
    static_assert(PM == 4 || PM == 8 || PM % 16 == 0, "C of 4 or 8 rows fills the first rows of one row tile, else whole tiles");
    constexpr bool HALF = PM < 16;          // rows PM..15 of the tile are zero and are not stored
    constexpr int MT = HALF ? 1 : PM / 16, KT = RB / 8;
    const int g = lane >> 2, t = lane & 3;
    const bool rowok = !HALF || g < PM;     // this lane's first row exists
    Tf32Pair a[MT][KT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int kt = 0; kt < KT; ++kt) {
            a[mt][kt][0] = tt_split_tf32(rowok ? Cs[(16 * mt + g) * CS + 8 * kt + t] : 0.f);
            a[mt][kt][2] = tt_split_tf32(rowok ? Cs[(16 * mt + g) * CS + 8 * kt + t + 4] : 0.f);
            if (HALF) {
                a[mt][kt][1].hi = 0u; a[mt][kt][1].lo = 0u; a[mt][kt][3].hi = 0u; a[mt][kt][3].lo = 0u;
            } else {
                a[mt][kt][1] = tt_split_tf32(Cs[(16 * mt + g + 8) * CS + 8 * kt + t]);
                a[mt][kt][3] = tt_split_tf32(Cs[(16 * mt + g + 8) * CS + 8 * kt + t + 4]);
            }
        }
    const int K = w.K;
    const float* __restrict__ GK = td.core[K - 1];
    const uint32_t* __restrict__ rows = w.val[K];
    const int rb_ = g >> 2, jb = g & 3;   // this lane's B-fragment column: child row rb_ of the pair, output column jb
    const int rc = t >> 1, jc = 2 * (t & 1);  // this lane's C-fragment columns: child row rc, output columns jc, jc+1
    constexpr int NP = MT == 1 ? 3 : 2;   // row pairs in flight (two where C has two row tiles: registers)
    constexpr uint32_t IDC = 32 - 32 % (2 * NP);   // rows per id chunk: a multiple of the rows per iteration
    uint32_t ids = 0, cb = u0;   // last digits of IDC rows at a time, one per lane (the loop takes them by shuffle)
    for (uint32_t ub = u0; ub < u1; ub += 2 * NP) {
        if (ub == cb + IDC || ub == u0) {
            cb = ub;
            ids = (lane < IDC && ub + lane < u1) ? rows[ub + lane] - row_base : 0u;
        }
        float bv[NP][KT][2];
#pragma unroll
        for (int np = 0; np < NP; ++np) {
            // an odd tail (or a missing second pair) repeats the last row; it is computed but not stored
            const uint32_t ul = min(ub + 2 * np + (uint32_t)rb_, u1 - 1);
            const uint32_t iK = __shfl_sync(0xffffffffu, ids, ul - cb);
            const float* __restrict__ Dl = GK + (size_t)iK * (RB * 4) + jb;
#pragma unroll
            for (int kt = 0; kt < KT; ++kt) {
                bv[np][kt][0] = __ldg(Dl + (8 * kt + t) * 4);
                bv[np][kt][1] = __ldg(Dl + (8 * kt + t + 4) * 4);
            }
        }
#pragma unroll
        for (int np = 0; np < NP; ++np) {
            float acc[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) { acc[mt][0] = 0.f; acc[mt][1] = 0.f; acc[mt][2] = 0.f; acc[mt][3] = 0.f; }
#pragma unroll
            for (int kt = 0; kt < KT; ++kt) {
                Tf32Pair b[2];
                b[0] = tt_split_tf32(bv[np][kt][0]);
                b[1] = tt_split_tf32(bv[np][kt][1]);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) tt_mma_3xtf32(acc[mt], a[mt][kt], b);
            }
            const uint32_t us = ub + 2 * np + (uint32_t)rc;
            if (us < u1) {
                float* e = w.E + (size_t)us * (PM * 4) + jc;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    if (rowok) __stcs(reinterpret_cast<float2*>(e + (16 * mt + g) * 4), make_float2(acc[mt][0], acc[mt][1]));
                    if (!HALF) __stcs(reinterpret_cast<float2*>(e + (16 * mt + g + 8) * 4), make_float2(acc[mt][2], acc[mt][3]));
                }
            }
        }
    }
}

// The same product for C of 8 or 4 rows (d_1 d_2 = 8 or 4), where the form above fills half or a quarter of its row
// tile: transposed, E_u[p][j] = sum_b D_u[b][j] * C[p][b] as m16n8k8 tiles with M = 16 = four child rows x 4 columns
// j, K = 8 values of b, N = 8 rows p of C (PM = 4: columns 4..7 are zero operands).  Half the tensor-core
// instructions per row (a quarter for PM = 4); the split fragments of C^T take RB/2 registers.  A lane ends up with
// single floats of four rows of E (p = 2t, 2t+1; column j = g % 4) and stores them as such.
template <int PM, int RB, int CS = RB>
__device__ __forceinline__ void tt_warp_rows_mma_t(const float* Cs, const WsView& w, const TableDesc& td, uint32_t u0, uint32_t u1,
                                                   uint32_t row_base, int lane)
{
    static_assert(PM == 8 || PM == 4, "C of 8 or 4 rows");
    constexpr int KT = RB / 8;
    const int g = lane >> 2, t = lane & 3;
    const bool pok = g < PM;                // this lane's column p of C^T exists
    Tf32Pair cb[KT][2];                     // B[k = b][n = p] = C[p][b]
#pragma unroll
    for (int kt = 0; kt < KT; ++kt) {
        cb[kt][0] = tt_split_tf32(pok ? Cs[g * CS + 8 * kt + t] : 0.f);
        cb[kt][1] = tt_split_tf32(pok ? Cs[g * CS + 8 * kt + t + 4] : 0.f);
    }
    const int K = w.K;
    const float* __restrict__ GK = td.core[K - 1];
    const uint32_t* __restrict__ rows = w.val[K];
    const int q0 = g >> 2, j = g & 3;       // A-fragment rows g and g + 8: child rows q0 and q0 + 2 of the four, column j
    constexpr int NQ = 2;                   // fours of rows in flight
    constexpr uint32_t IDC = 32;            // rows per id chunk: a multiple of the rows per iteration
    uint32_t ids = 0, cbase = u0;           // last digits of IDC rows at a time, one per lane (the loop takes them by shuffle)
    for (uint32_t ub = u0; ub < u1; ub += 4 * NQ) {
        if (ub == cbase + IDC || ub == u0) {
            cbase = ub;
            ids = (ub + lane < u1) ? rows[ub + lane] - row_base : 0u;
        }
        float av[NQ][KT][4];
#pragma unroll
        for (int nq = 0; nq < NQ; ++nq) {
            // a short tail repeats the last row; it is computed but not stored
            const uint32_t ula = min(ub + 4 * nq + (uint32_t)q0, u1 - 1), ulc = min(ub + 4 * nq + (uint32_t)q0 + 2, u1 - 1);
            const uint32_t iKa = __shfl_sync(0xffffffffu, ids, ula - cbase), iKc = __shfl_sync(0xffffffffu, ids, ulc - cbase);
            const float* __restrict__ Da = GK + (size_t)iKa * (RB * 4) + j;
            const float* __restrict__ Dc = GK + (size_t)iKc * (RB * 4) + j;
#pragma unroll
            for (int kt = 0; kt < KT; ++kt) {
                av[nq][kt][0] = __ldg(Da + (8 * kt + t) * 4);
                av[nq][kt][1] = __ldg(Dc + (8 * kt + t) * 4);
                av[nq][kt][2] = __ldg(Da + (8 * kt + t + 4) * 4);
                av[nq][kt][3] = __ldg(Dc + (8 * kt + t + 4) * 4);
            }
        }
#pragma unroll
        for (int nq = 0; nq < NQ; ++nq) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kt = 0; kt < KT; ++kt) {
                Tf32Pair a[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) a[x] = tt_split_tf32(av[nq][kt][x]);
                tt_mma_3xtf32(acc, a, cb[kt]);
            }
            // acc: E[p = 2t][j], E[2t + 1][j] of child row q0, then of child row q0 + 2
            const uint32_t usa = ub + 4 * nq + (uint32_t)q0, usc = usa + 2;
            if (2 * t < PM) {
                if (usa < u1) {
                    float* e = w.E + (size_t)usa * (PM * 4) + (2 * t) * 4 + j;
                    __stcs(e, acc[0]);
                    __stcs(e + 4, acc[1]);
                }
                if (usc < u1) {
                    float* e = w.E + (size_t)usc * (PM * 4) + (2 * t) * 4 + j;
                    __stcs(e, acc[2]);
                    __stcs(e + 4, acc[3]);
                }
            }
        }
    }
}

// one warp: groups fetched dynamically from the CTA's range through a shared counter
template <int PM, int RB, int TP, int M, int CPL, bool MMA>
__device__ __forceinline__ void tt_sweep_fast(const WsView& w, const TableDesc& td, uint32_t g1, float* As, float* Cs,
                                              uint32_t* next, int lane)
{
    const int K = w.K, km = K - 2;
    const int ra = td.r[km], cols = td.d[km] * RB;
    const uint32_t nK = (uint32_t)td.n[K - 1];
    for (;;) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(next, 1u);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= g1) break;
        if (!(w.ablation & 1)) g = w.tnode[K - 1][g];   // position in the digit-major order -> group
        const uint32_t val = w.val[K - 1][g];
        const float* src = tt_left_operand(w, td, K - 1, g);
        for (int i = lane; i < M * ra; i += 32) {
            const int m = i / ra, a = i - m * ra;
            As[a * M + m] = __ldg(src + i);
        }
        __syncwarp();
        const uint32_t im = val % (uint32_t)td.n[km];
        tt_warp_mid<M, CPL>(As, td.core[km] + (size_t)im * td.slice_floats[km], Cs, ra, cols, lane);
        __syncwarp();
        if constexpr (MMA) tt_warp_rows_mma<PM, RB>(Cs, w, td, w.cstart[K - 1][g], w.cstart[K - 1][g + 1], val * nK, lane);
        else tt_warp_rows<PM, RB, TP>(Cs, w, td, w.cstart[K - 1][g], w.cstart[K - 1][g + 1], val * nK, lane);
        __syncwarp();
    }
}

// Tensor-core variants: a warp takes NG = 16 / MROWS consecutive groups of the digit-major order at a time; their
// intermediate products are formed together (quad_mid.cuh), then each group's rows are produced from its C in shared
// memory, on the tensor cores too.
template <int PM, int RB, int MROWS, int KTMAX, bool FEW>
__device__ __forceinline__ void tt_sweep_quad(const WsView& w, const TableDesc& td, uint32_t g1, float* Cs4, uint32_t* next, int lane)
{
    constexpr int COLS = PM / MROWS * RB;   // d_{K-1} * r_{K-1}
    constexpr int NG = 16 / MROWS;
    const int K = w.K, km = K - 2;
    const int ra = td.r[km];
    const uint32_t nK = (uint32_t)td.n[K - 1];
    for (;;) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(next, FEW ? next[1] : (uint32_t)NG);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= g1) break;
        const int cnt = (int)min(FEW ? next[1] : (uint32_t)NG, g1 - base);
        uint32_t valq = 0, imq = 0, u0q = 0, u1q = 0;
        const float* srcq = nullptr;
        if (lane < cnt) {
            const uint32_t pos = base + lane;
            const uint32_t gq = (w.ablation & 1) ? pos : w.tnode[K - 1][pos];   // position in the digit-major order -> group
            valq = w.val[K - 1][gq];
            imq = valq % (uint32_t)td.n[km];
            srcq = tt_left_operand(w, td, K - 1, gq);
            u0q = w.cstart[K - 1][gq];
            u1q = w.cstart[K - 1][gq + 1];
        }
        tt_quad_mid<COLS, MROWS, KTMAX, RB>(td.core[km], td.slice_floats[km], ra, cnt, imq, srcq, Cs4, lane);
        __syncwarp();
        for (int q = 0; q < cnt; ++q) {
            const uint32_t val = __shfl_sync(0xffffffffu, valq, q);
            const uint32_t u0 = __shfl_sync(0xffffffffu, u0q, q), u1 = __shfl_sync(0xffffffffu, u1q, q);
            if constexpr (PM < 16) tt_warp_rows_mma_t<PM, RB, RB + 4>(Cs4 + (size_t)q * (PM * (RB + 4)), w, td, u0, u1, val * nK, lane);
            else tt_warp_rows_mma<PM, RB, RB + 4>(Cs4 + (size_t)q * (PM * (RB + 4)), w, td, u0, u1, val * nK, lane);
        }
        __syncwarp();
    }
}

// rank-64 four-core shape (wide.cuh): a warp makes one row, a lane one of its 32 rows of C by the four columns of the slice
template <bool FEW>
__global__ void __launch_bounds__(WIDE_THREADS, 2) k_sweep_fwd_wide(WsView w, int vbase)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ WideBatch batches[2];
    float *Bs = sm, *As = Bs + 64 * WIDE_BP, *Cs = As + 8 * WIDE_GROUPS * WIDE_AP;
    const int t = w.vlist[vbase + (FEW ? blockIdx.x : blockIdx.y)], K = w.K, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const TableDesc& td = w.tdesc[t];
    uint32_t step;
    const uint2 rng = tt_sweep_unit<FEW>(w, t, WIDE_GROUPS, step);
    const uint32_t nK = (uint32_t)td.n[K - 1];
    WideLoop<false> loop(w, td, rng, batches, Bs, As, Cs);
    while (loop.next()) {
        const WideBatch& b = loop.batch();
        const uint32_t rows = wide_rows(b);
        float4* stage = reinterpret_cast<float4*>(As) + wid * 64;   // this warp's slices of the last core, one at a time
        for (uint32_t r = wid; r < rows; r += WIDE_THREADS / 32) {
            uint32_t u;
            const int q = wide_row(b, r, u);
            const float4* D = reinterpret_cast<const float4*>(td.core[K - 1]) + (size_t)(w.val[K][u] - b.val[q] * nK) * 64;
            __syncwarp();
            tt_cp_async16(stage + lane, D + lane);
            tt_cp_async16(stage + lane + 32, D + lane + 32);
            asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            const float4* c4 = reinterpret_cast<const float4*>(Cs + q * (32 * WIDE_CP) + lane * WIDE_CP);
            float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int i = 0; i < 16; ++i) {
                const float4 c = c4[i];
                const float4 d0 = stage[4 * i], d1 = stage[4 * i + 1], d2 = stage[4 * i + 2], d3 = stage[4 * i + 3];
                e.x = fmaf(c.x, d0.x, e.x); e.y = fmaf(c.x, d0.y, e.y); e.z = fmaf(c.x, d0.z, e.z); e.w = fmaf(c.x, d0.w, e.w);
                e.x = fmaf(c.y, d1.x, e.x); e.y = fmaf(c.y, d1.y, e.y); e.z = fmaf(c.y, d1.z, e.z); e.w = fmaf(c.y, d1.w, e.w);
                e.x = fmaf(c.z, d2.x, e.x); e.y = fmaf(c.z, d2.y, e.y); e.z = fmaf(c.z, d2.z, e.z); e.w = fmaf(c.z, d2.w, e.w);
                e.x = fmaf(c.w, d3.x, e.x); e.y = fmaf(c.w, d3.y, e.y); e.z = fmaf(c.w, d3.z, e.z); e.w = fmaf(c.w, d3.w, e.w);
            }
            reinterpret_cast<float4*>(w.E + (size_t)u * w.D)[lane] = e;
        }
    }
}

// any shape: batches of groups spread flat over the CTA (generic.cuh)
__global__ void __launch_bounds__(GEN_THREADS) k_sweep_fwd_any(WsView w, int vbase)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ GenBatch b;
    const int t = w.vlist[vbase + blockIdx.y];
    const uint2 rng = w.unit_rng[t * w.units_per_table + blockIdx.x];
    const TableDesc& td = w.tdesc[t];
    const bool vec = (td.d[w.K - 1] & 3) == 0;   // then slices, their rows and the row buffer's rows are whole float4s
    const uint32_t ng = (uint32_t)gen_groups(td, w.K);
    uint2 groups, range;
    gen_unit(w, t, rng, groups, range);
    for (uint32_t base = groups.x; base < groups.y; base += ng) {
        const int cnt = (int)min(ng, groups.y - base);
        gen_batch_begin(w, td, base, cnt, range, b);
        gen_batch_c<GEN_THREADS>(w, td, cnt, b, sm);
        const uint32_t rows = b.row0[cnt];
        for (uint32_t r0 = 0; r0 < rows; r0 += GEN_ROWS) {
            const int n = (int)min((uint32_t)GEN_ROWS, rows - r0);
            gen_rows(w, td, cnt, r0, n, b);
            if (vec) gen_forward_rows<true>(w, td, n, b, sm);
            else gen_forward_rows<false>(w, td, n, b, sm);
            __syncthreads();
        }
        __syncthreads();
    }
}

// fused levels K-1 and K: C stays on chip, rows go to w.E.  One CTA (4 warps) per work unit (table, q);
// one instantiation per shape variant V so that each gets its own register budget.  blockIdx.y walks the
// tables of variant V (w.vlist), blockIdx.x the table's equal-cost slices.
template <int V, bool FEW>
__global__ void __launch_bounds__(128, V != 3 ? 6 : 1) k_sweep_fwd(WsView w, int pl_floats, int c_floats, int vbase)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ uint32_t next[2];   // the CTA's next group, groups that a warp takes at a time
    const int t = w.vlist[vbase + (FEW ? blockIdx.x : blockIdx.y)];
    uint32_t step;
    const uint2 rng = tt_sweep_unit<FEW>(w, t, V < 5 ? 4 : 8, step);
    const uint32_t g1 = rng.y;
    const TableDesc& td = w.tdesc[t];
    if (threadIdx.x == 0) { next[0] = rng.x; next[1] = step; }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (V == 0) tt_sweep_quad<16, 32, 4, 4, FEW>(w, td, g1, sm + (size_t)wid * (4 * 16 * 36), next, lane);
    if (V == 1) tt_sweep_quad<16, 16, 4, 4, FEW>(w, td, g1, sm + (size_t)wid * (4 * 16 * 20), next, lane);
    if (V == 3) tt_sweep_quad<32, 32, 4, 4, FEW>(w, td, g1, sm + (size_t)wid * (4 * 32 * 36), next, lane);
    float* As = sm + (size_t)wid * (pl_floats + c_floats);
    float* Cs = As + pl_floats;
    if (V == 2) tt_sweep_quad<16, 8, 4, 4, FEW>(w, td, g1, sm + (size_t)wid * (4 * 16 * 12), next, lane);
    if (V == 5) tt_sweep_quad<8, 32, 2, 4, FEW>(w, td, g1, sm + (size_t)wid * (8 * 8 * 36), next, lane);
    if (V == 6) tt_sweep_quad<8, 16, 2, 4, FEW>(w, td, g1, sm + (size_t)wid * (8 * 8 * 20), next, lane);
    if (V == 7) tt_sweep_quad<8, 8, 2, 4, FEW>(w, td, g1, sm + (size_t)wid * (8 * 8 * 12), next, lane);
    if (V == 8) tt_sweep_quad<4, 32, 2, 4, FEW>(w, td, g1, sm + (size_t)wid * (8 * 4 * 36), next, lane);
    if (V == 9) tt_sweep_quad<4, 16, 2, 4, FEW>(w, td, g1, sm + (size_t)wid * (8 * 4 * 20), next, lane);
    if (V == 10) tt_sweep_fast<4, 8, 2, 2, 1, false>(w, td, g1, As, Cs, next, lane);
}

// dynamic shared memory of k_sweep_fwd<V> / k_sweep_bwd<V>: four C tiles per warp for the tensor-core variants
static size_t tt_sweep_smem(int V, int max_pl, int max_c)
{
    if (V == 0) return (size_t)4 * 4 * 16 * 36 * sizeof(float);   // C rows padded by four floats (conflict-free fragment loads)
    if (V == 1) return (size_t)4 * 4 * 16 * 20 * sizeof(float);
    if (V == 3) return (size_t)4 * 4 * 32 * 36 * sizeof(float);
    if (V == 5) return (size_t)4 * 8 * 8 * 36 * sizeof(float);    // eight C tiles of 8 rows per warp
    if (V == 6) return (size_t)4 * 8 * 8 * 20 * sizeof(float);
    if (V == 2) return (size_t)4 * 4 * 16 * 12 * sizeof(float);
    if (V == 7) return (size_t)4 * 8 * 8 * 12 * sizeof(float);
    if (V == 8) return (size_t)4 * 8 * 4 * 36 * sizeof(float);
    if (V == 9) return (size_t)4 * 8 * 4 * 20 * sizeof(float);
    return (size_t)4 * (max_pl + max_c) * sizeof(float);
}

template <int V>
static cudaError_t launch_sweep_fwd(tt_emb* h, int max_pl, int max_c, cudaStream_t s)
{
    const int n = h->vcount[V + 1];
    if (n == 0) return cudaSuccess;
    [[maybe_unused]] const bool few = tt_few_groups(h);
    cudaError_t e;
    if ((e = tt_stage_begin(h, 9 + V + 1, s)) != cudaSuccess) return e;
    if constexpr (V < 0) {
        const size_t smem = GEN_C_FLOATS * sizeof(float);
        if ((e = cudaFuncSetAttribute(k_sweep_fwd_any, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(k_sweep_fwd_any, dim3(h->units_per_table, n), dim3(GEN_THREADS), smem, s, h->v, h->vbase[0])) != cudaSuccess) return e;
    } else if constexpr (V == 4) {
        auto kern = few ? k_sweep_fwd_wide<true> : k_sweep_fwd_wide<false>;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WIDE_SMEM)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(kern, few ? dim3(n, h->sweep_ctas) : dim3(h->units_per_table, n), dim3(WIDE_THREADS), WIDE_SMEM, s, h->v, h->vbase[V + 1])) != cudaSuccess) return e;
    } else {
        const size_t smem = tt_sweep_smem(V, max_pl, max_c);
        auto kern = few ? k_sweep_fwd<V, true> : k_sweep_fwd<V, false>;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(kern, few ? dim3(n, h->sweep_ctas) : dim3(h->units_per_table, n), dim3(128), smem, s, h->v, max_pl, max_c, h->vbase[V + 1])) != cudaSuccess) return e;
    }
    tt_note_launch();
    if ((e = tt_stage_end(h, 9 + V + 1, s)) != cudaSuccess) return e;
    return cudaGetLastError();
}

// Whether level 2 is multiplied digit by digit.  k_level2 starts CTAs for every i_2 and looks at every possible prefix; a node
// by itself costs a read of its slice.  Forward call by node / by digit, us: n = 64^4, rank 64, 131 k lookups 238 / 201; n =
// (1 M, 8, 8, 8), rank 64, 1 k lookups (8 k possible prefixes per lookup) 529 / 595, 131 k (61) 3760 / 2547; n = (4096, 4096,
// 8, 8), rank 64, 131 k (128) 1456 / 1559 and 6553 / 4155 (popular and spread rows), rank 9 952 / 1063 and 1360 / 1598; n = (8,
// 1 M, 8, 8), 131 k lookups (an eighth of a node per slice) 596 / 2320.
#define LEVEL2_PER_SLICE 4
#define LEVEL2_SPARSE 64
static bool tt_level2_by_digit(const tt_emb* h)
{
    const WsView& w = h->v;
    if (w.ablation & 1) return false;
    const uint64_t nodes = w.L < (int64_t)w.cap[2] ? (uint64_t)w.L : w.cap[2];   // at most
    uint64_t slices = 0, space = 0;
    for (int t = 0; t < h->T; ++t) {
        slices += (uint64_t)h->tab[t].n[1];
        space += h->tab[t].prefix_space[2];
    }
    return nodes >= LEVEL2_PER_SLICE * slices && space <= LEVEL2_SPARSE * nodes;
}

cudaError_t tt_launch_contraction(tt_emb* h, cudaStream_t s)
{
    WsView& w = h->v;
    int max_pl = 4, max_c = 4;
    for (int t = 0; t < h->T; ++t) {
        const TableDesc& td = h->tab[t];
        for (int k = 1; k < h->K; ++k) {
            int f = (td.P[k] * td.r[k] + 3) / 4 * 4;
            if (k <= h->K - 2 && f > max_pl) max_pl = f;
            if (k == h->K - 1 && f > max_c) max_c = f;
        }
    }
    cudaError_t e;
    if (h->K == 4 && tt_level2_by_digit(h)) {
        uint32_t max_x = 1, max_z = 1;
        for (int t = 0; t < h->T; ++t) {
            const TableDesc& td = h->tab[t];
            const uint32_t x = (uint32_t)td.n[1] * tt_level2_parts(td), z = (uint32_t)((td.d[1] * td.r[2] + MT_EDGE - 1) / MT_EDGE);
            if (x > max_x) max_x = x;
            if (z > max_z) max_z = z;
        }
        if ((e = tt_launch_pdl(k_level2, dim3(max_x, h->T, max_z), dim3(128), 0, s, w)) != cudaSuccess) return e;
        tt_note_launch();
    } else if (h->K == 4) {
        if ((e = tt_launch_pdl(k_level2_nodes, dim3(h->sm_count * 16), dim3(128), (size_t)max_pl * sizeof(float), s, w)) != cudaSuccess) return e;
        tt_note_launch();
    }
    // tables of different shape variants are independent: their kernels run side by side on forked streams
    int nvar = 0;
    for (int vi = 0; vi <= TT_NUM_VARIANTS; ++vi) nvar += h->vcount[vi] > 0 ? 1 : 0;
    const bool fork = nvar > 1 && !h->serial;
    if (fork && (e = tt_fork(h, s, 4)) != cudaSuccess) return e;
    int slot = 0;
    auto next_stream = [&](int vi) { return (fork && h->vcount[vi] > 0) ? h->side[(slot++) & 3] : s; };
    if ((e = launch_sweep_fwd<-1>(h, max_pl, max_c, next_stream(0))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<0>(h, max_pl, max_c, next_stream(1))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<1>(h, max_pl, max_c, next_stream(2))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<2>(h, max_pl, max_c, next_stream(3))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<3>(h, max_pl, max_c, next_stream(4))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<4>(h, max_pl, max_c, next_stream(5))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<5>(h, max_pl, max_c, next_stream(6))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<6>(h, max_pl, max_c, next_stream(7))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<7>(h, max_pl, max_c, next_stream(8))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<8>(h, max_pl, max_c, next_stream(9))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<9>(h, max_pl, max_c, next_stream(10))) != cudaSuccess) return e;
    if ((e = launch_sweep_fwd<10>(h, max_pl, max_c, next_stream(11))) != cudaSuccess) return e;
    if (fork && (e = tt_join(h, s, 4)) != cudaSuccess) return e;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- pooling

// One warp per bag.  A row of D floats is read as D/4 float4 chunks by a sub-warp of LPR lanes
// (LPR = power of two >= min(32, D/4)); 32/LPR rows are fetched per load instruction, up to NF such
// instructions are issued back to back before any result is consumed (the kernel is bound by memory
// latency, so bytes in flight per warp are what counts), the rank look-ups of the next 32 lookups are
// started before the current ones are gathered, and the sub-warps' partial sums are combined with
// __shfl_xor at the end.
__device__ __forceinline__ uint32_t tt_lookup_slot(const WsView& w, const TableDesc& td, int64_t l, uint32_t capK)
{
    const int64_t g = tt_index<true>(w, l);    // streamed once: evict-first, keeps L2 for rows and rank words
    uint32_t slot = 0xffffffffu;
    if (w.ablation & 4) return (g >= 0 && g < td.N && l < (int64_t)capK) ? (uint32_t)l : slot;   // no de-duplication: lookup l is row slot l
    if (g >= 0 && g < td.N) {
        const uint2 e = __ldg(&w.bm[td.word_base + ((uint32_t)g >> 5)]);
        if (e.x >> (g & 31) & 1u) {
            slot = e.y + __popc(e.x & ((1u << (g & 31)) - 1u));
            if (slot >= capK) slot = 0xffffffffu;
        }
    }
    return slot;
}

// Pooling partition: the lookups are cut into C = W * chunks equal shares of whole bags (boundaries: group.cuh), and the
// warps take the shares in order from a counter.  All resident warps therefore work inside one moving window of
// about W shares at a time - a few tables - so the rows that several bags share are still in L2 when the next
// bag asks for them; one contiguous share per warp would spread the warps over all tables at once.  Equal lookups are
// not equal time (a share of popular rows is served by L2, one of unpopular rows by HBM): with a fixed assignment the
// first warp finished at 84 % of the kernel, the median one at 90 %.  Eight shares per warp: more of them cost more
// in pipeline fill and drain per share than they give in balance (4 / 8 / 16 / 32: 2.62 / 2.39 / 2.50 / 2.76 ms).
#define TT_POOL_MAX_CHUNKS 8
// grid and shares of a pooling kernel with W warps
static void tt_pool_set(tt_emb* h, int64_t grid, int warps)
{
    const int64_t W = grid * warps;
    int64_t c = h->v.L / (W * 512);                     // at least 512 lookups per share
    c = c < 1 ? 1 : (c > TT_POOL_MAX_CHUNKS ? TT_POOL_MAX_CHUNKS : c);
    while (W * c > TT_POOL_MAX_SHARES && c > 1) --c;
    h->pool_grid = (int)grid;
    h->v.pool_shares = W * c;
}

template <int LPR, int CPL, bool WT>  // lanes per row, float4 chunks per lane, weighted / mean pooling
__global__ void __launch_bounds__(256, (CPL == 1 ? 6 : (CPL == 2 ? 2 : 1))) k_pool_vec(WsView w, float* __restrict__ out)
{
    tt_pdl_enter();
    const int lane = threadIdx.x & 31;
    const int sub = lane / LPR, lr = lane % LPR;
    constexpr int RPI = 32 / LPR;                       // rows per load instruction
    constexpr int NIT = 32 / RPI;                       // load instructions per 32 lookups
    constexpr int NF = NIT < 4 ? NIT : 4;               // load instructions in flight
    const int D4 = w.D >> 2;
    const float4* __restrict__ E4 = reinterpret_cast<const float4*>(w.E);
    const uint32_t capK = w.cap[w.K];
    // Skew-aware split: the grid is exactly resident (persistent warps); a share holds the bags whose first
    // lookup falls into it (offsets is the cost prefix sum).
    const int64_t C = w.pool_shares;
    auto clampL = [&](int64_t x) { return x < 0 ? (int64_t)0 : (x > w.L ? w.L : x); };
    for (;;) {
    // shares are handed out in order through a counter: a warp whose shares hold popular (L2-resident) rows takes more of them
    int64_t ci = 0;
    if (lane == 0) ci = (int64_t)atomicAdd(&w.counters[CTR_POOL_NEXT], 1u);
    ci = __shfl_sync(0xffffffffu, ci, 0);
    if (ci >= C) break;
    const int64_t b0 = __ldg(w.pool_bounds + ci), b1 = __ldg(w.pool_bounds + ci + 1);
    if (b0 >= b1) continue;
    // every bag is summed over its own (offsets[bag], offsets[bag + 1]) pair, clamped to [0, L]; an inverted pair (malformed
    // offsets) is an empty bag.  o_next: start of the next bag = this bag's end as stored, before the inversion fix
    int64_t o_lo = clampL(__ldg(w.offsets + b0)), o_next = clampL(__ldg(w.offsets + b0 + 1));
    int64_t o_hi = o_next < o_lo ? o_lo : o_next;
    int t = (int)(b0 / w.B);
    uint32_t slot_next;
    float wt_next = 1.f;
    auto fetch = [&](int64_t base, int64_t lim, int tt) {   // rank look-up (and weight) of lookup base + lane
        slot_next = (base + lane < lim) ? tt_lookup_slot(w, w.tdesc[tt], base + lane, capK) : 0xffffffffu;
        if (WT) wt_next = (w.psw && base + lane < lim) ? __ldg(w.psw + base + lane) : 1.f;
    };
    fetch(o_lo, o_hi, t);
    for (int64_t bag = b0; bag < b1; ++bag) {
        const int64_t b = bag - (int64_t)t * w.B;
        // next bag (for the prefetch of its first 32 rank look-ups)
        const bool has_next = bag + 1 < b1;
        const int64_t n_lo = o_next;
        const int64_t n_next = has_next ? clampL(__ldg(w.offsets + bag + 2)) : o_next;
        const int64_t n_hi = n_next < n_lo ? n_lo : n_next;
        const int tn = (has_next && b + 1 == w.B) ? t + 1 : t;
        float4 acc[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (o_lo >= o_hi && has_next) fetch(n_lo, n_hi, tn);
        for (int64_t l0 = o_lo; l0 < o_hi; l0 += 32) {
            const uint32_t slot = slot_next;
            const float wt = wt_next;
            if (w.upairs && l0 + lane < o_hi) __stcs(&w.upairs[l0 + lane], make_uint2(slot, (uint32_t)b));  // kept for the backward sort
            if (l0 + 32 < o_hi) fetch(l0 + 32, o_hi, t);
            else if (has_next) fetch(n_lo, n_hi, tn);
            const int n = (int)min((int64_t)32, o_hi - l0);
            float4 part[CPL];   // two-level sum: per-batch partial, added to the bag's sum once per batch
#pragma unroll
            for (int c = 0; c < CPL; ++c) part[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j0 = 0; j0 < NIT; j0 += NF) {
                if (j0 * RPI >= n) break;
                float4 v[NF][CPL];
#pragma unroll
                for (int jj = 0; jj < NF; ++jj) {
                    const int j = (j0 + jj) * RPI + sub;
                    const uint32_t sl = __shfl_sync(0xffffffffu, slot, j & 31);
                    const bool ok = j < n && sl != 0xffffffffu;
                    const float4* row = E4 + (size_t)(ok ? sl : 0u) * D4;
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        const int ch = lr + c * LPR;
                        v[jj][c] = (ok && ch < D4) ? __ldg(row + ch) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
#pragma unroll
                for (int jj = 0; jj < NF; ++jj) {
                    const float wj = WT ? __shfl_sync(0xffffffffu, wt, ((j0 + jj) * RPI + sub) & 31) : 1.f;
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        if (WT) {
                            part[c].x = fmaf(wj, v[jj][c].x, part[c].x); part[c].y = fmaf(wj, v[jj][c].y, part[c].y);
                            part[c].z = fmaf(wj, v[jj][c].z, part[c].z); part[c].w = fmaf(wj, v[jj][c].w, part[c].w);
                        } else {
                            part[c].x += v[jj][c].x; part[c].y += v[jj][c].y; part[c].z += v[jj][c].z; part[c].w += v[jj][c].w;
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < CPL; ++c) { acc[c].x += part[c].x; acc[c].y += part[c].y; acc[c].z += part[c].z; acc[c].w += part[c].w; }
        }
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, o);
                acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, o);
                acc[c].z += __shfl_xor_sync(0xffffffffu, acc[c].z, o);
                acc[c].w += __shfl_xor_sync(0xffffffffu, acc[c].w, o);
            }
        }
        if (sub == 0) {
            float4* o4 = reinterpret_cast<float4*>(out + (size_t)b * w.T * w.D + (size_t)t * w.D);
            const float inv = (WT && w.pool_mean && o_hi > o_lo) ? 1.f / (float)(o_hi - o_lo) : 1.f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int ch = lr + c * LPR;
                if (WT) { acc[c].x *= inv; acc[c].y *= inv; acc[c].z *= inv; acc[c].w *= inv; }
                if (ch < D4) __stcs(o4 + ch, acc[c]);
            }
        }
        o_lo = n_lo;
        o_hi = n_hi;
        o_next = n_next;
        t = tn;
    }
    }
}

// Rows of up to 256 bytes (D <= 64): the gather is bound by bytes in flight, and registers cap what LDG can keep in
// flight.  Here every warp owns an 8 KB shared-memory buffer and fills it with cp.async (16 bytes per lane, two
// rows per instruction, no staging registers): the 32 rows of a batch are all in flight at once.  Same bag
// partition (equal shares of the lookups per warp), same prefetch of the next batch's rank look-ups.
#define POOL_WARPS 7   // 4 CTAs x 7 warps x 8 KB = 224 KB of the SM's shared memory
template <int R4, bool WT>   // R4: float4 pieces per staged row, 16 (D <= 64) or 8 (D <= 32)
__global__ void __launch_bounds__(32 * POOL_WARPS, 4) k_pool_async(WsView w, float* __restrict__ out)
{
    tt_pdl_enter();
    static_assert(R4 == 16 || R4 == 8, "two or four rows per cp.async instruction");
    constexpr int RPI = 32 / R4;
    constexpr int PGRP = 4;              // load instructions per group: a window is cut short and tested for validity per group
                                         // (half of all windows end a bag and are short; groups of two measured slower)
    extern __shared__ __align__(16) float4 pool_buf[];   // [POOL_WARPS][32 rows][R4 float4]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int sub = lane / R4, lr = lane % R4;
    float4* buf = pool_buf + (size_t)wid * 32 * R4;
    const int D4 = w.D >> 2;
    const bool lane_on = lr < D4;
    const float4* __restrict__ E4 = reinterpret_cast<const float4*>(w.E);
    const uint32_t capK = w.cap[w.K];
    const int64_t C = w.pool_shares;
    // lookup positions and bag indices fit in 32 bits (L and T * B are below 2^31, checked when the handle is made)
    typedef int32_t pos_t;
    auto clampL = [&](int64_t x) { return x < 0 ? (pos_t)0 : (x > w.L ? (pos_t)w.L : (pos_t)x); };
    for (;;) {
    // shares are handed out in order through a counter: a warp whose shares hold popular (L2-resident) rows takes more of them
    int64_t ci = 0;
    if (lane == 0) ci = (int64_t)atomicAdd(&w.counters[CTR_POOL_NEXT], 1u);
    ci = __shfl_sync(0xffffffffu, ci, 0);
    if (ci >= C) break;
    const pos_t b0 = (pos_t)__ldg(w.pool_bounds + ci), b1 = (pos_t)__ldg(w.pool_bounds + ci + 1);
    if (b0 >= b1) continue;
    // every bag is summed over its own (offsets[bag], offsets[bag + 1]) pair, clamped to [0, L]; an inverted pair (malformed
    // offsets) is an empty bag.  o_next: start of the next bag = this bag's end as stored, before the inversion fix
    pos_t o_lo = clampL(__ldg(w.offsets + b0)), o_next = clampL(__ldg(w.offsets + b0 + 1));
    pos_t o_hi = o_next < o_lo ? o_lo : o_next;
    int t = (int)(b0 / w.B);
    uint32_t slot_next;
    float wt_next = 1.f;
    auto fetch = [&](pos_t base, pos_t lim, int tt) {   // rank look-up (and weight) of lookup base + lane
        slot_next = (base + lane < lim) ? tt_lookup_slot(w, w.tdesc[tt], base + lane, capK) : 0xffffffffu;
        if (WT) wt_next = (w.psw && base + lane < lim) ? __ldg(w.psw + base + lane) : 1.f;
    };
    fetch(o_lo, o_hi, t);
    for (pos_t bag = b0; bag < b1; ++bag) {
        const pos_t b = bag - (pos_t)t * w.B;
        const bool has_next = bag + 1 < b1;
        const pos_t n_lo = o_next;
        const pos_t n_next = has_next ? clampL(__ldg(w.offsets + bag + 2)) : o_next;
        const pos_t n_hi = n_next < n_lo ? n_lo : n_next;
        const int tn = (has_next && b + 1 == w.B) ? t + 1 : t;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (o_lo >= o_hi && has_next) fetch(n_lo, n_hi, tn);
        for (pos_t l0 = o_lo; l0 < o_hi; l0 += 32) {
            const uint32_t slot = slot_next;
            const float wt = wt_next;
            if (w.upairs && l0 + lane < o_hi) __stcs(&w.upairs[l0 + lane], make_uint2(slot, (uint32_t)b));
            const int n = (int)min((pos_t)32, o_hi - l0);
            const unsigned valid = __ballot_sync(0xffffffffu, lane < n && slot != 0xffffffffu);
            // two-level sum: the batch's rows go into a partial that is added to the bag's sum once per batch, so the
            // rounding error of a bag with thousands of lookups grows with the number of batches, not of rows
            float4 part = make_float4(0.f, 0.f, 0.f, 0.f);
            // all rows of the batch in flight
            // (groups of four instructions; a short window -- half of all windows end a bag -- leaves early)
            // a group whose rows are all valid (the usual case) needs no per-row test
            const bool plain = valid == (n == 32 ? 0xffffffffu : (1u << n) - 1u) && D4 == R4;
#pragma unroll
            for (int jq = 0; jq < 32 / RPI; jq += PGRP) {
                if (RPI * jq >= n) break;
                if (plain && RPI * (jq + PGRP) <= n) {
#pragma unroll
                    for (int jj = jq; jj < jq + PGRP; ++jj) {
                        const int j = RPI * jj + sub;
                        const uint32_t sl = __shfl_sync(0xffffffffu, slot, j);
                        tt_cp_async16(buf + j * R4 + lr, E4 + (size_t)sl * R4 + lr);
                    }
                } else {
#pragma unroll
                    for (int jj = jq; jj < jq + PGRP; ++jj) {
                        const int j = RPI * jj + sub;
                        const uint32_t sl = __shfl_sync(0xffffffffu, slot, j);
                        if (((valid >> j) & 1u) && lane_on) tt_cp_async16(buf + j * R4 + lr, E4 + (size_t)sl * D4 + lr);
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            // the rank look-ups of the next batch (or of the next bag) overlap the gather
            if (l0 + 32 < o_hi) fetch(l0 + 32, o_hi, t);
            else if (has_next) fetch(n_lo, n_hi, tn);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
#pragma unroll
            for (int jq = 0; jq < 32 / RPI; jq += PGRP) {
                if (RPI * jq >= n) break;
                if (!WT && plain && RPI * (jq + PGRP) <= n) {
#pragma unroll
                    for (int jj = jq; jj < jq + PGRP; ++jj) {
                        const float4 v = buf[(RPI * jj + sub) * R4 + lr];
                        tt_add4(part, v);
                    }
                } else {
#pragma unroll
                    for (int jj = jq; jj < jq + PGRP; ++jj) {
                        const int j = RPI * jj + sub;
                        const float wj = WT ? __shfl_sync(0xffffffffu, wt, j) : 1.f;
                        if (((valid >> j) & 1u) && lane_on) {
                            const float4 v = buf[j * R4 + lr];
                            if (WT) { part.x = fmaf(wj, v.x, part.x); part.y = fmaf(wj, v.y, part.y); part.z = fmaf(wj, v.z, part.z); part.w = fmaf(wj, v.w, part.w); }
                            else tt_add4(part, v);
                        }
                    }
                }
            }
            acc.x += part.x; acc.y += part.y; acc.z += part.z; acc.w += part.w;
            __syncwarp();
        }
#pragma unroll
        for (int o = R4; o < 32; o <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        }
        if (WT && w.pool_mean && o_hi > o_lo) {
            const float inv = 1.f / (float)(o_hi - o_lo);
            acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
        }
        if (sub == 0 && lane_on) __stcs(reinterpret_cast<float4*>(out + (size_t)b * w.T * w.D + (size_t)t * w.D) + lr, acc);
        o_lo = n_lo;
        o_hi = n_hi;
        o_next = n_next;
        t = tn;
    }
    }
}

// The same gather for batches with few lookups per bag (on average below TT_POOL_STREAM_BELOW, or ..._WIDE for rows
// of more than 128 bytes): a window is 32 consecutive lookups of the warp's share, whatever bags they belong to.  One
// bag per window, as in k_pool_async, costs the latency of a window per bag: 2 million bags took 0.82 ms there whether
// they held 2 or 16 lookups each, and 7.9 million one-lookup bags 3.0 ms.  Here a window of one-lookup bags goes
// straight from the staged rows to out (those 7.9 million bags: 0.40 ms, 5 TB/s of rows read and written); a full
// window with one boundary is summed into two partial sums in one unrolled pass; a window with several bags in it is
// summed by the whole warp at once, each sub-warp taking consecutive rows and the pieces of a bag that crosses
// sub-warps being joined afterwards (from two boundaries on for rows of up to 128 bytes, from five on for wider rows,
// where a sub-warp has sixteen rows to walk); a window with empty bags in it deals its bags out to the sub-warps.  Weights and
// mean pooling take the same ways (the factor with the row, 1 / length where a bag is written): 131 k bags of 1 to 30 weighted
// rows of 128 bytes 73 -> 63 us, of 1 to 8 rows of 256 bytes with mean 51 -> 41 us, of one weighted row 33 -> 17 us against
// bag by bag.
// 2 million bags of 128-byte rows, stream against one bag per window: 2 / 4 / 8 lookups each 0.20 / 0.28 / 0.51 ms against 0.82; 1
// to 15 lookups 0.54 against 0.83, 1 to 31 0.83 against 0.91, 1 to 63 1.22 against 1.27, 1 to 100 1.69 against 1.72, 1 to 200 3.09
// against 3.00 ms; 262 k bags of 0 to 4 rows, mean, 67 us bag by bag, 34 with the bags dealt out.  256-byte rows: 2 / 4 / 8 lookups
// 0.29 / 0.44 / 0.74 ms against 0.88-0.92; 1 to 15 lookups 0.78 against 0.95; 1 to 31 1.11-1.19 against 1.10; on the benchmark
// configuration (1 to 100 lookups) 2.34-2.36 against 2.39 ms.  Hence the thresholds (the benchmark configuration stays with the
// per-bag kernel).  A window ends early only at the end of the share or of a table (the rank look-up of a window uses one table).
// With malformed offsets (status bit set by the offsets check earlier in the stream) every bag is summed over its own clamped
// (offsets[bag], offsets[bag + 1]) pair as the header promises, and windows stop at the end of their bag.
#define TT_POOL_STREAM_BELOW 33        // rows of up to 128 bytes
#define TT_POOL_STREAM_BELOW_WIDE 12   // rows of up to 256 bytes
// a += v, or a += f * v with weights
template <bool WT>
__device__ __forceinline__ void pool_add(float4& a, const float4& v, float f)
{
    if (WT) a = make_float4(fmaf(f, v.x, a.x), fmaf(f, v.y, a.y), fmaf(f, v.z, a.z), fmaf(f, v.w, a.w));
    else tt_add4(a, v);
}

template <int R4, bool WT>   // R4: float4 pieces per staged row, 16 (D <= 64) or 8 (D <= 32)
__global__ void __launch_bounds__(32 * POOL_WARPS, 4) k_pool_stream(WsView w, float* __restrict__ out)
{
    tt_pdl_enter();
    static_assert(R4 == 16 || R4 == 8, "two or four rows per cp.async instruction");
    constexpr int RPI = 32 / R4;
    constexpr int PGRP = 4;              // load instructions per group: a window is cut short and tested for validity per group
    extern __shared__ __align__(16) float4 pool_buf[];   // [POOL_WARPS][32 rows][R4 float4]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int sub = lane / R4, lr = lane % R4;
    float4* buf = pool_buf + (size_t)wid * 32 * R4;
    const int D4 = w.D >> 2;
    const bool lane_on = lr < D4;
    const float4* __restrict__ E4 = reinterpret_cast<const float4*>(w.E);
    const uint32_t capK = w.cap[w.K];
    const int64_t C = w.pool_shares;
    const bool stream_ok = !(*w.status & TT_EMB_STATUS_OFFSETS);
    // lookup positions and bag indices fit in 32 bits (L and T * B are below 2^31, checked when the handle is made)
    typedef int32_t pos_t;
    auto clampL = [&](int64_t x) { return x < 0 ? (pos_t)0 : (x > w.L ? (pos_t)w.L : (pos_t)x); };
    for (;;) {
    int64_t ci = 0;     // shares are handed out in order through a counter (see k_pool_async)
    if (lane == 0) ci = (int64_t)atomicAdd(&w.counters[CTR_POOL_NEXT], 1u);
    ci = __shfl_sync(0xffffffffu, ci, 0);
    if (ci >= C) break;
    const pos_t b0 = (pos_t)__ldg(w.pool_bounds + ci), b1 = (pos_t)__ldg(w.pool_bounds + ci + 1);
    if (b0 >= b1) continue;
    // the ends of the share's bags, 32 at a time and one vector ahead: lane i holds the clamped offsets[ebase + 1 + i]
    // (ends_nx: the 32 bags after those), so that no bag waits for a load of its own end
    auto load_ends = [&](pos_t base) { const pos_t i = base + lane; return i < b1 ? clampL(__ldg(w.offsets + i + 1)) : (pos_t)0x7fffffff; };   // past the share: never inside a window
    pos_t ebase = b0;
    pos_t ends_reg = load_ends(b0), ends_nx = load_ends(b0 + 32);
    auto end_of = [&](pos_t bg) {     // bg >= ebase, and below ebase + 64 (a step moves on by at most 32 bags)
        while (bg - ebase >= 32) {
            ends_reg = ends_nx;
            ebase += 32;
            ends_nx = load_ends(ebase + 32);
        }
        return __shfl_sync(0xffffffffu, ends_reg, (int)(bg - ebase));
    };
    // the bag being summed: its table, its (clamped) range, the end of the bag as stored
    pos_t bag = b0;
    int t = (int)(b0 / w.B);
    pos_t o_lo = clampL(__ldg(w.offsets + b0)), o_next = end_of(b0);
    pos_t o_hi = o_next < o_lo ? o_lo : o_next;
    const pos_t share_end = stream_ok ? clampL(__ldg(w.offsets + b1)) : 0;
    pos_t t_end = stream_ok ? (pos_t)__ldg(w.tl_start + t + 1) : 0;
    pos_t pos = o_lo;                                 // next lookup of the stream
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    // rank look-up (and weight) of lookup base + lane, for the window that starts at `base`
    uint32_t slot_next = 0xffffffffu;
    float wt_next = 1.f;
    pos_t pre_pos = -1;
    int pre_t = -1;
    auto fetch = [&](pos_t base, pos_t lim, int tt) {
        slot_next = (base + lane < lim) ? tt_lookup_slot(w, w.tdesc[tt], base + lane, capK) : 0xffffffffu;
        if (WT) wt_next = (w.psw && base + lane < lim) ? __ldg(w.psw + base + lane) : 1.f;
        pre_pos = base;
        pre_t = tt;
    };
    // bag `nb_`, which starts at lookup `lo_`, becomes the one being summed (nb_ > bag, at most 32 bags on)
    auto seek_bag = [&](pos_t nb_, pos_t lo_) {
        acc = make_float4(0.f, 0.f, 0.f, 0.f);
        bag = nb_;
        if (bag < b1) {
            if (bag >= (pos_t)(t + 1) * w.B) {
                ++t;
                if (stream_ok) t_end = (pos_t)__ldg(w.tl_start + t + 1);
            }
            o_lo = lo_;
            o_next = end_of(bag);
            o_hi = o_next < o_lo ? o_lo : o_next;
        }
    };
    auto advance_bag = [&]() { seek_bag(bag + 1, o_next); };
    // the bag is complete: combine the sub-warps, write its row of out, move on to the next bag
    auto close_bag = [&]() {
#pragma unroll
        for (int o = R4; o < 32; o <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        }
        if (WT && w.pool_mean && o_hi > o_lo) {
            const float inv = 1.f / (float)(o_hi - o_lo);
            acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
        }
        const pos_t b = bag - (pos_t)t * w.B;
        if (sub == 0 && lane_on) __stcs(reinterpret_cast<float4*>(out + (size_t)b * w.T * w.D + (size_t)t * w.D) + lr, acc);
        advance_bag();
    };
    while (bag < b1) {
        if (pos >= o_hi) {              // the bag has no (more) lookups
            close_bag();
            pos = o_lo;
            continue;
        }
        const pos_t lim = stream_ok ? (share_end < t_end ? share_end : t_end) : o_hi;   // > pos: the bag ends no later
        const int n = (int)min((pos_t)32, lim - pos);
        if (pre_pos != pos || pre_t != t) fetch(pos, lim, t);
        const uint32_t slot = slot_next;
        const float wt = wt_next;
        const unsigned valid = __ballot_sync(0xffffffffu, lane < n && slot != 0xffffffffu);
        // all rows of the window in flight (groups of four instructions; a short window leaves early);
        // a group whose rows are all valid (the usual case) needs no per-row test
        const bool plain = valid == (n == 32 ? 0xffffffffu : (1u << n) - 1u) && D4 == R4;
#pragma unroll
        for (int jq = 0; jq < 32 / RPI; jq += PGRP) {
            if (RPI * jq >= n) break;
            if (plain && RPI * (jq + PGRP) <= n) {
#pragma unroll
                for (int jj = jq; jj < jq + PGRP; ++jj) {
                    const int j = RPI * jj + sub;
                    const uint32_t sl = __shfl_sync(0xffffffffu, slot, j);
                    tt_cp_async16(buf + j * R4 + lr, E4 + (size_t)sl * R4 + lr);
                }
            } else {
#pragma unroll
                for (int jj = jq; jj < jq + PGRP; ++jj) {
                    const int j = RPI * jj + sub;
                    const uint32_t sl = __shfl_sync(0xffffffffu, slot, j);
                    if (((valid >> j) & 1u) && lane_on) tt_cp_async16(buf + j * R4 + lr, E4 + (size_t)sl * D4 + lr);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        // the rank look-ups of the next window overlap the gather (the next window of the stream; in the per-bag mode
        // only while the bag goes on)
        {
            const pos_t np = pos + n;
            if (stream_ok) {
                if (np < lim) fetch(np, lim, t);
                else if (np < share_end) {               // the table ends here: the next window belongs to the next one
                    const pos_t te = (pos_t)__ldg(w.tl_start + t + 2);
                    fetch(np, share_end < te ? share_end : te, t + 1);
                }
            } else if (np < o_hi) fetch(np, o_hi, t);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        // Windows with bag boundaries in them are summed by the whole warp at once.  Lane i looks at bag + i, which ends at
        // e_mine; a bag starts at row e - pos of the window for every end e inside it.
        if (stream_ok && o_hi < pos + n) {
            const pos_t wend = pos + n;
            const int ei = (int)(bag - ebase) + lane;
            const pos_t e0 = __shfl_sync(0xffffffffu, ends_reg, ei & 31), e1 = __shfl_sync(0xffffffffu, ends_nx, ei & 31);
            const pos_t e_mine = ei < 32 ? e0 : e1;
            // one-lookup bags only (lane i: bag + i ends at pos + i + 1): every staged row is a row of out
            if (o_lo == pos && __all_sync(0xffffffffu, lane >= n || e_mine == pos + lane + 1)) {
                const pos_t bf = bag - (pos_t)t * w.B;       // the window lies in table t: bf + n <= B
                if (w.upairs && lane < n) __stcs(&w.upairs[pos + lane], make_uint2(slot, (uint32_t)(bf + lane)));
                float4* o4 = reinterpret_cast<float4*>(out + (size_t)bf * w.T * w.D + (size_t)t * w.D) + lr;
                const size_t ostride = (size_t)w.T * D4;
#pragma unroll
                for (int jj = 0; jj < 32 / RPI; ++jj) {
                    const int j = RPI * jj + sub;
                    const float wj = WT ? __shfl_sync(0xffffffffu, wt, j) : 1.f;   // (the mean of one lookup is the lookup)
                    if (j < n && lane_on) {
                        float4 v = ((valid >> j) & 1u) ? buf[j * R4 + lr] : make_float4(0.f, 0.f, 0.f, 0.f);
                        if (WT) v = make_float4(wj * v.x, wj * v.y, wj * v.z, wj * v.w);
                        __stcs(o4 + (size_t)j * ostride, v);
                    }
                }
                __syncwarp();
                pos += n;
                seek_bag(bag + n, pos);
                continue;
            }
            const pos_t e_prev = __shfl_up_sync(0xffffffffu, e_mine, 1);
            // Empty bags among those that start inside the window: the bags that end in it and the one that goes on are dealt out to the
            // sub-warps, 32 at a time, an empty one as a sum of no rows.  Row r of a bag goes to partial sum r % RPI: as many partial
            // sums as where the sub-warps share a bag.  Bag by bag / dealt out, 131 k bags, us: 128-byte rows: half of the bags empty,
            // the others of 4, 10, 20 and 40 rows 33 / 21, 41 / 29, 49 / 41, 66 / 59 (weighted 35 / 22, 43 / 33, 54 / 47, 76 / 70), 30 %
            // empty, the others of 30 rows 68 / 63 (79 / 74); 256-byte rows: 35 / 27, 45 / 37, 61 / 53, 84 / 84 (39 / 29, 51 / 41, 70 / 61,
            // 93 / 92), 80 / 83 (86 / 86).  With at least 3, 5 or 9 bags in the window only: never faster, 43 / 50 at 20 rows with 5.
            const bool empties = __any_sync(0xffffffffu, lane >= 1 && e_prev < wend && e_mine == e_prev);
            if (empties) {
                const pos_t base = pos;
                const int t0 = t;
                for (pos_t e = e_mine;;) {
                    const int nc = __popc(__ballot_sync(0xffffffffu, e <= wend && bag + lane < (pos_t)(t + 1) * w.B));   // of this table
                    const pos_t ended = __shfl_sync(0xffffffffu, e, (nc - 1) & 31), last = nc > 0 ? ended : o_lo, upto = nc < 32 ? wend : last;
                    const int nb = nc + (last < upto ? 1 : 0);
                    const pos_t bt = bag - (pos_t)t * w.B;
                    if (w.upairs) {
                        int k = 0;          // bags that end before or at this lane's row
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1)
                            if (__shfl_sync(0xffffffffu, e, k + step - 1) <= base + lane) k += step;
                        if (base + lane >= pos && base + lane < upto) __stcs(&w.upairs[base + lane], make_uint2(slot, (uint32_t)(bt + k)));
                    }
                    float4 carry = acc;     // the open bag's sum so far, the same in every sub-warp
#pragma unroll
                    for (int o = R4; o < 32; o <<= 1) {
                        carry.x += __shfl_xor_sync(0xffffffffu, carry.x, o); carry.y += __shfl_xor_sync(0xffffffffu, carry.y, o);
                        carry.z += __shfl_xor_sync(0xffffffffu, carry.z, o); carry.w += __shfl_xor_sync(0xffffffffu, carry.w, o);
                    }
                    float4 keep = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int i0 = 0; i0 < nb; i0 += RPI) {
                        const int i = i0 + sub, ii = i < nb ? i : nb - 1;
                        const pos_t hi = __shfl_sync(0xffffffffu, e, ii & 31), before = __shfl_sync(0xffffffffu, e, (ii - 1) & 31);
                        const pos_t lo = ii > 0 ? before : o_lo;
                        const int j0 = (int)((lo > pos ? lo : pos) - base), len = i < nb ? (int)((hi < upto ? hi : upto) - base) - j0 : 0;
                        const int steps = __reduce_max_sync(0xffffffffu, (len + RPI - 1) / RPI);   // (weights come by shuffle)
                        unsigned rows = len > 0 ? (valid >> j0) & (0xffffffffu >> (32 - len)) : 0u;
                        const float4* src = buf + j0 * R4 + lr;
                        float4 part[RPI];
#pragma unroll
                        for (int c = 0; c < RPI; ++c) part[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                        for (int st = 0; st < steps; ++st, rows >>= RPI, src += RPI * R4) {
#pragma unroll
                            for (int c = 0; c < RPI; ++c) {
                                const float wj = WT ? __shfl_sync(0xffffffffu, wt, (j0 + st * RPI + c) & 31) : 1.f;
                                if (rows & (1u << c)) pool_add<WT>(part[c], src[c * R4], wj);
                            }
                        }
#pragma unroll
                        for (int o = 1; o < RPI; o <<= 1)
#pragma unroll
                            for (int c = 0; c < RPI; c += 2 * o) tt_add4(part[c], part[c + o]);
                        float4 sum = part[0];
                        if (i >= nb || !lane_on) continue;
                        if (i == 0) tt_add4(sum, carry);
                        if (i >= nc) { keep = sum; continue; }
                        if (WT && w.pool_mean && hi > lo) {
                            const float inv = 1.f / (float)(hi - lo);
                            sum = make_float4(sum.x * inv, sum.y * inv, sum.z * inv, sum.w * inv);
                        }
                        __stcs(reinterpret_cast<float4*>(out + (size_t)(bt + i) * w.T * w.D + (size_t)t * w.D) + lr, sum);
                    }
                    pos = upto;
                    seek_bag(bag + nc, last);
                    acc = keep;
                    if (nc < 32 || bag >= b1 || t != t0) break;
                    const int ei = (int)(bag - ebase) + lane;
                    const pos_t x0 = __shfl_sync(0xffffffffu, ends_reg, ei & 31), x1 = __shfl_sync(0xffffffffu, ends_nx, ei & 31);
                    e = ei < 32 ? x0 : x1;
                }
                __syncwarp();
                continue;
            }
            const int inside = __popc(__ballot_sync(0xffffffffu, e_mine > pos && e_mine < wend));   // bag ends inside the window
            if (inside == 1 && plain && n == 32) {
                // one boundary, at row c: the rows before it complete the open bag, the others start the next one
                const int c = (int)(o_hi - pos);
                if (w.upairs) __stcs(&w.upairs[pos + lane], make_uint2(slot, (uint32_t)(bag - (pos_t)t * w.B) + (lane >= c ? 1u : 0u)));
                float4 pa = make_float4(0.f, 0.f, 0.f, 0.f), pb = pa;
#pragma unroll
                for (int jj = 0; jj < 32 / RPI; ++jj) {
                    const int j = RPI * jj + sub;
                    const float4 v = buf[j * R4 + lr];
                    const float wj = WT ? __shfl_sync(0xffffffffu, wt, j) : 1.f;
                    if (j < c) pool_add<WT>(pa, v, wj); else pool_add<WT>(pb, v, wj);
                }
                acc.x += pa.x; acc.y += pa.y; acc.z += pa.z; acc.w += pa.w;
                close_bag();
                acc = pb;
                __syncwarp();
                pos = wend;
                continue;
            }
            const bool many = inside >= (R4 == 16 ? 5 : 2);   // fewer: cheaper bag by bag
            if (many) {
                // starts: bit j = row j is the first of its bag; closes: bit j = row j is the last of its bag
                const unsigned starts = __reduce_or_sync(0xffffffffu, (e_mine > pos && e_mine < wend) ? 1u << (int)(e_mine - pos) : 0u)
                                      | (o_lo == pos ? 1u : 0u);
                const bool last_closed = __any_sync(0xffffffffu, e_mine == wend);
                const unsigned closes = (starts >> 1) | (last_closed ? 1u << (n - 1) : 0u);
                const pos_t bt = bag - (pos_t)t * w.B;       // bag of row j: bt + bags started in rows 1..j
                auto row_of = [&](int j) {
                    const pos_t b = bt + __popc(starts & ((2u << j) - 2u));
                    return reinterpret_cast<float4*>(out + (size_t)b * w.T * w.D + (size_t)t * w.D) + lr;
                };
                if (w.upairs && lane < n)
                    __stcs(&w.upairs[pos + lane], make_uint2(slot, (uint32_t)(bt + __popc(starts & ((2u << lane) - 2u)))));
                // the open bag's sum so far, the same in every sub-warp
                float4 carry = acc;
#pragma unroll
                for (int o = R4; o < 32; o <<= 1) {
                    carry.x += __shfl_xor_sync(0xffffffffu, carry.x, o); carry.y += __shfl_xor_sync(0xffffffffu, carry.y, o);
                    carry.z += __shfl_xor_sync(0xffffffffu, carry.z, o); carry.w += __shfl_xor_sync(0xffffffffu, carry.w, o);
                }
                // sub-warp s sums the R4 consecutive rows from s * R4 on, in step with the others: a bag that lies inside
                // them is written at its last row; the piece of a bag that came in from before (head) is kept, the piece
                // of a bag that goes on after them is what `run` holds at the end
                float4 run = make_float4(0.f, 0.f, 0.f, 0.f), head = run;
                bool head_open = !((starts >> (sub * R4)) & 1u), head_closed = false;
                // (not unrolled: the kernel's warps are spread over its four summing paths, and with this loop unrolled
                // they waited for instructions: 2.39 -> 1.90 ms on the 240-table workload, ncu `no_instruction` stalls)
                // (the row of out of the bag being summed moves on by one bag per segment end; masks shifted to the sub-warp)
                {
                    // (weights come by shuffle: then all sub-warps take the same number of steps, and those past the window's
                    // last row do nothing)
                    const int j0 = sub * R4, ns = min(R4, WT ? n : n - j0);
                    int len = 0;                                  // rows of the running bag, for the mean
                    unsigned vs = valid >> j0, cs = closes >> j0;
                    float4* orow = row_of(j0);
                    const size_t ostride = (size_t)w.T * D4;
                    const float4* src = buf + j0 * R4 + lr;
#pragma unroll 1
                    for (int jj = 0; jj < ns; ++jj, vs >>= 1, cs >>= 1, src += R4) {
                        const float wj = WT ? __shfl_sync(0xffffffffu, wt, j0 + jj) : 1.f;
                        if (vs & 1u) {
                            const float4 v = *src;
                            pool_add<WT>(run, v, wj);
                        }
                        if (WT) ++len;
                        if (cs & 1u) {
                            if (head_open) { head = run; head_closed = true; head_open = false; }
                            else if (lane_on) {
                                if (WT && w.pool_mean) {
                                    const float inv = 1.f / (float)len;
                                    run = make_float4(run.x * inv, run.y * inv, run.z * inv, run.w * inv);
                                }
                                __stcs(orow, run);
                            }
                            if (WT) len = 0;
                            run = make_float4(0.f, 0.f, 0.f, 0.f);
                            orow += ostride;
                        }
                    }
                }
                // the pieces across the sub-warps, in order: a head closes the bag carried so far; rows that all belong to
                // the carried bag add to it; otherwise the carried bag ended with the sub-warp before (nothing carried)
                const unsigned hc = __ballot_sync(0xffffffffu, head_closed), ho = __ballot_sync(0xffffffffu, head_open);
#pragma unroll
                for (int s2 = 0; s2 < RPI; ++s2) {
                    float inv = 1.f;
                    if (WT && w.pool_mean) {   // the bag that is open at the sub-warp's first row: bag + kb
                        const int kb = __popc(starts & ((2u << (s2 * R4)) - 2u));
                        const pos_t e_end = __shfl_sync(0xffffffffu, e_mine, kb), e_beg = __shfl_sync(0xffffffffu, e_mine, kb > 0 ? kb - 1 : 0);
                        inv = 1.f / (float)(e_end - (kb > 0 ? e_beg : o_lo));
                    }
                    if (((hc >> (s2 * R4)) & 1u) && sub == s2 && lane_on) {
                        float4 sum = carry;
                        tt_add4(sum, head);
                        if (WT && w.pool_mean) sum = make_float4(sum.x * inv, sum.y * inv, sum.z * inv, sum.w * inv);
                        __stcs(row_of(s2 * R4), sum);
                    }
                    float4 tail;
                    tail.x = __shfl_sync(0xffffffffu, run.x, s2 * R4 + lr); tail.y = __shfl_sync(0xffffffffu, run.y, s2 * R4 + lr);
                    tail.z = __shfl_sync(0xffffffffu, run.z, s2 * R4 + lr); tail.w = __shfl_sync(0xffffffffu, run.w, s2 * R4 + lr);
                    if ((ho >> (s2 * R4)) & 1u) tt_add4(carry, tail);
                    else carry = tail;
                }
                __syncwarp();
                const pos_t bl = bag + __popc(starts & 0xfffffffeu);     // the bag of the window's last row
                pos = wend;
                if (last_closed) seek_bag(bl + 1, pos);
                else {
                    if (bl > bag) {
                        const pos_t lo_ = end_of(bl - 1);
                        seek_bag(bl, lo_);
                    }
                    acc = sub == 0 ? carry : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                continue;
            }
        }
        // the window's rows, bag by bag.  Two-level sum: the rows of a (piece of a) bag go into a partial that is added to
        // the bag's sum once, so the rounding error of a bag with thousands of lookups grows with the number of windows
        int r = 0;
        while (r < n) {
            if (pos + r >= o_hi) {       // a bag ends inside the window (and empty bags after it)
                close_bag();
                if (bag >= b1) break;    // cannot happen with checked offsets; never spin on it
                continue;
            }
            const pos_t room = o_hi - (pos + r);
            const int seg = room < (pos_t)(n - r) ? (int)room : n - r;
            if (w.upairs && lane >= r && lane < r + seg)    // kept for the backward sort
                __stcs(&w.upairs[pos + lane], make_uint2(slot, (uint32_t)(bag - (pos_t)t * w.B)));
            if (!WT && seg == 1 && pos + r == o_lo && o_hi - o_lo == 1) {
                // a bag of one lookup: its row of out is the staged row (or zeros for an id outside the table); the
                // sub-warp that staged it writes it, nothing to combine
                if (sub == (r & (RPI - 1)) && lane_on) {
                    const float4 v = ((valid >> r) & 1u) ? buf[r * R4 + lr] : make_float4(0.f, 0.f, 0.f, 0.f);
                    __stcs(reinterpret_cast<float4*>(out + (size_t)(bag - (pos_t)t * w.B) * w.T * w.D + (size_t)t * w.D) + lr, v);
                }
                advance_bag();
                r += 1;
                if (bag >= b1) break;
                continue;
            }
            float4 part = make_float4(0.f, 0.f, 0.f, 0.f);
            if (plain && seg == 32) {
#pragma unroll
                for (int jj = 0; jj < 32 / RPI; ++jj) {
                    const float4 v = buf[(RPI * jj + sub) * R4 + lr];
                    pool_add<WT>(part, v, WT ? __shfl_sync(0xffffffffu, wt, RPI * jj + sub) : 1.f);
                }
            } else {
                for (int jj = r / RPI; RPI * jj < r + seg; ++jj) {
                    const int j = RPI * jj + sub;
                    const float wj = WT ? __shfl_sync(0xffffffffu, wt, j) : 1.f;
                    if (j >= r && j < r + seg && ((valid >> j) & 1u) && lane_on) {
                        const float4 v = buf[j * R4 + lr];
                        if (WT) { part.x = fmaf(wj, v.x, part.x); part.y = fmaf(wj, v.y, part.y); part.z = fmaf(wj, v.z, part.z); part.w = fmaf(wj, v.w, part.w); }
                        else tt_add4(part, v);
                    }
                }
            }
            acc.x += part.x; acc.y += part.y; acc.z += part.z; acc.w += part.w;
            r += seg;
        }
        __syncwarp();
        pos += n;
    }
    }
}


template <int R4, bool WT>
static cudaError_t launch_pool_async(tt_emb* h, float* out, bool plan, cudaStream_t s)
{
    const size_t smem = (size_t)POOL_WARPS * 32 * R4 * sizeof(float4);
    cudaError_t e = cudaFuncSetAttribute(k_pool_async<R4, WT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t nb = (int64_t)h->v.T * h->v.B;
    if (plan) {
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pool_async<R4, WT>, 32 * POOL_WARPS, smem)) != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        int64_t grid = (int64_t)per_sm * h->sm_count;
        const int64_t need = (nb + POOL_WARPS - 1) / POOL_WARPS;
        if (grid > need) grid = need;
        if (grid < 1) grid = 1;
        tt_pool_set(h, grid, POOL_WARPS);
        return cudaSuccess;
    }
    const int grid = h->pool_grid;
    if (h->v.L < (int64_t)(R4 == 16 ? TT_POOL_STREAM_BELOW_WIDE : TT_POOL_STREAM_BELOW) * nb) {   // few lookups per bag: windows across bags
        if ((e = cudaFuncSetAttribute(k_pool_stream<R4, WT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(k_pool_stream<R4, WT>, dim3(grid), dim3(32 * POOL_WARPS), smem, s, h->v, out)) != cudaSuccess) return e;
        tt_note_launch();
        return cudaGetLastError();
    }
    if ((e = tt_launch_pdl(k_pool_async<R4, WT>, dim3(grid), dim3(32 * POOL_WARPS), smem, s, h->v, out)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

template <int LPR, int CPL, bool WT>
static cudaError_t launch_pool_vec(tt_emb* h, float* out, bool plan, cudaStream_t s)
{
    cudaError_t e;
    if (plan) {
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pool_vec<LPR, CPL, WT>, 256, 0)) != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        const int64_t nb = (int64_t)h->v.T * h->v.B;
        int64_t grid = (int64_t)per_sm * h->sm_count;
        const int64_t need = (nb + 7) / 8;
        if (grid > need) grid = need;
        if (grid < 1) grid = 1;
        tt_pool_set(h, grid, 8);
        return cudaSuccess;
    }
    if ((e = tt_launch_pdl(k_pool_vec<LPR, CPL, WT>, dim3(h->pool_grid), dim3(256), 0, s, h->v, out)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

// Rows whose length is no multiple of four floats (or an `out` that is not 16-byte aligned), D <= 4 R4 - 3: a row starts anywhere
// in its first 16-byte piece, so the R4 or fewer aligned pieces that it touches are staged as they lie and every lane picks its
// columns (lane, lane + 32) behind the row's shift.  Same shares, windows and look-ahead as k_pool_async; the pieces past the last row
// of the row buffer lie in its guard bytes.  1 M lookups of 45 floats: 101 us with a row per pair of 4-byte loads and a warp per bag,
// 66 us now (2.7 TB/s of rows; the window's chain row id -> rank word -> rows, as in k_pool_async).
template <int R4, bool WT>
__global__ void __launch_bounds__(32 * POOL_WARPS, 4) k_pool_odd(WsView w, float* __restrict__ out)
{
    tt_pdl_enter();
    static_assert(R4 == 16 || R4 == 8, "two or four rows per cp.async instruction");
    constexpr int RPI = 32 / R4, P = 4 * R4;             // pitch of a staged row in floats
    extern __shared__ __align__(16) float4 pool_buf[];   // [POOL_WARPS][32 rows][R4 float4]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int sub = lane / R4, lr = lane % R4;
    float4* buf = pool_buf + (size_t)wid * 32 * R4;
    const float* bufv = reinterpret_cast<const float*>(buf);
    const uint32_t D = (uint32_t)w.D;
    const bool on0 = lane < (int)D, on1 = R4 == 16 && lane + 32 < (int)D;
    const uint32_t capK = w.cap[w.K];
    const int64_t C = w.pool_shares;
    typedef int32_t pos_t;
    auto clampL = [&](int64_t x) { return x < 0 ? (pos_t)0 : (x > w.L ? (pos_t)w.L : (pos_t)x); };
    for (;;) {
    int64_t ci = 0;     // shares are handed out in order through a counter (see k_pool_async)
    if (lane == 0) ci = (int64_t)atomicAdd(&w.counters[CTR_POOL_NEXT], 1u);
    ci = __shfl_sync(0xffffffffu, ci, 0);
    if (ci >= C) break;
    const pos_t b0 = (pos_t)__ldg(w.pool_bounds + ci), b1 = (pos_t)__ldg(w.pool_bounds + ci + 1);
    if (b0 >= b1) continue;
    pos_t o_lo = clampL(__ldg(w.offsets + b0)), o_next = clampL(__ldg(w.offsets + b0 + 1));
    pos_t o_hi = o_next < o_lo ? o_lo : o_next;
    int t = (int)(b0 / w.B);
    uint32_t slot_next;
    float wt_next = 1.f;
    auto fetch = [&](pos_t base, pos_t lim, int tt) {   // rank look-up (and weight) of lookup base + lane
        slot_next = (base + lane < lim) ? tt_lookup_slot(w, w.tdesc[tt], base + lane, capK) : 0xffffffffu;
        if (WT) wt_next = (w.psw && base + lane < lim) ? __ldg(w.psw + base + lane) : 1.f;
    };
    fetch(o_lo, o_hi, t);
    for (pos_t bag = b0; bag < b1; ++bag) {
        const pos_t b = bag - (pos_t)t * w.B;
        const bool has_next = bag + 1 < b1;
        const pos_t n_lo = o_next;
        const pos_t n_next = has_next ? clampL(__ldg(w.offsets + bag + 2)) : o_next;
        const pos_t n_hi = n_next < n_lo ? n_lo : n_next;
        const int tn = (has_next && b + 1 == w.B) ? t + 1 : t;
        float acc0 = 0.f, acc1 = 0.f;
        if (o_lo >= o_hi && has_next) fetch(n_lo, n_hi, tn);
        for (pos_t l0 = o_lo; l0 < o_hi; l0 += 32) {
            const uint32_t slot = slot_next;
            const float wt = wt_next;
            if (w.upairs && l0 + lane < o_hi) __stcs(&w.upairs[l0 + lane], make_uint2(slot, (uint32_t)b));
            const int n = (int)min((pos_t)32, o_hi - l0);
            const unsigned valid = __ballot_sync(0xffffffffu, lane < n && slot != 0xffffffffu);
#pragma unroll 4
            for (int jq = 0; jq < 32 / RPI; ++jq) {
                if (RPI * jq >= n) break;
                const int j = RPI * jq + sub;
                const uint32_t sl = __shfl_sync(0xffffffffu, slot, j);
                const uint64_t start = (uint64_t)sl * D;
                if (((valid >> j) & 1u) && 4u * lr < (uint32_t)(start & 3) + D) tt_cp_async16(buf + j * R4 + lr, w.E + (start & ~(uint64_t)3) + 4 * lr);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            // the rank look-ups of the next batch (or of the next bag) overlap the gather
            if (l0 + 32 < o_hi) fetch(l0 + 32, o_hi, t);
            else if (has_next) fetch(n_lo, n_hi, tn);
            const uint32_t shift = (slot * D) & 3u;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            float part0 = 0.f, part1 = 0.f;   // two-level sum: added to the bag's sum once per batch
            for (int j0 = 0; j0 < n; j0 += 8) {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) {
                    const int j = j0 + jj;
                    const float* src = bufv + j * P + __shfl_sync(0xffffffffu, shift, j) + lane;
                    const float wj = WT ? __shfl_sync(0xffffffffu, wt, j) : 1.f;
                    const bool ok = (valid >> j) & 1u;
                    const float x0 = ok && on0 ? src[0] : 0.f;
                    part0 = WT ? fmaf(wj, x0, part0) : part0 + x0;
                    if (R4 == 16) {
                        const float x1 = ok && on1 ? src[32] : 0.f;
                        part1 = WT ? fmaf(wj, x1, part1) : part1 + x1;
                    }
                }
            }
            acc0 += part0;
            acc1 += part1;
            __syncwarp();
        }
        if (WT && w.pool_mean && o_hi > o_lo) {
            const float inv = 1.f / (float)(o_hi - o_lo);
            acc0 *= inv;
            acc1 *= inv;
        }
        float* o = out + ((size_t)b * w.T + t) * D + lane;
        if (on0) __stcs(o, acc0);
        if (on1) __stcs(o + 32, acc1);
        o_lo = n_lo;
        o_hi = n_hi;
        o_next = n_next;
        t = tn;
    }
    }
}

template <int R4, bool WT>
static cudaError_t launch_pool_odd(tt_emb* h, float* out, bool plan, cudaStream_t s)
{
    const size_t smem = (size_t)POOL_WARPS * 32 * R4 * sizeof(float4);
    cudaError_t e = cudaFuncSetAttribute(k_pool_odd<R4, WT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (plan) {
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pool_odd<R4, WT>, 32 * POOL_WARPS, smem)) != cudaSuccess) return e;
        const int64_t need = ((int64_t)h->v.T * h->v.B + POOL_WARPS - 1) / POOL_WARPS, most = (int64_t)(per_sm < 1 ? 1 : per_sm) * h->sm_count;
        tt_pool_set(h, need < 1 ? 1 : (need < most ? need : most), POOL_WARPS);
        return cudaSuccess;
    }
    if ((e = tt_launch_pdl(k_pool_odd<R4, WT>, dim3(h->pool_grid), dim3(32 * POOL_WARPS), smem, s, h->v, out)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

// any D (scalar path): lane handles elements lane, lane + 32, ... (NC of them per pass over the bag); 32 / NC rows in flight
template <int NC>
__global__ void __launch_bounds__(256) k_pool_scalar(WsView w, float* __restrict__ out)
{
    tt_pdl_enter();
    constexpr int RF = 32 / NC;     // rows in flight
    const int lane = threadIdx.x & 31;
    const int D = w.D;
    const int64_t nb = (int64_t)w.T * w.B;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t capK = w.cap[w.K];
    for (int64_t bag = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); bag < nb; bag += nwarps) {
        const int t = (int)(bag / w.B);
        const int64_t b = bag - (int64_t)t * w.B;
        const TableDesc& td = w.tdesc[t];
        int64_t lo = w.offsets[bag], hi = w.offsets[bag + 1];
        lo = lo < 0 ? 0 : (lo > w.L ? w.L : lo);
        hi = hi < lo ? lo : (hi > w.L ? w.L : hi);
        float* o = out + (size_t)b * w.T * D + (size_t)t * D;
        for (int e0 = 0; e0 < D; e0 += 32 * NC) {
            float acc[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = 0.f;
            // 32 lookups at a time: every lane looks one slot up (the two dependent loads of a lookup run 32 wide instead of
            // one after the other), then the rows are added in lookup order, RF row loads in flight
            for (int64_t l0 = lo; l0 < hi; l0 += 32) {
                const int n = (int)min((int64_t)32, hi - l0);
                const uint32_t slot = lane < n ? tt_lookup_slot(w, td, l0 + lane, capK) : 0xffffffffu;
                const float a = (w.psw && lane < n) ? __ldg(w.psw + l0 + lane) : 1.f;
                if (w.upairs && e0 == 0 && lane < n) w.upairs[l0 + lane] = make_uint2(slot, (uint32_t)b);
                for (int j0 = 0; j0 < n; j0 += RF) {
                    float v[RF][NC], aj[RF];
#pragma unroll
                    for (int jj = 0; jj < RF; ++jj) {
                        const uint32_t sj = __shfl_sync(0xffffffffu, slot, (j0 + jj) & 31);
                        aj[jj] = __shfl_sync(0xffffffffu, a, (j0 + jj) & 31);
                        const bool ok = j0 + jj < n && sj != 0xffffffffu;
                        const float* row = w.E + (size_t)(ok ? sj : 0u) * D;
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const int idx = e0 + lane + c * 32;
                            v[jj][c] = (ok && idx < D) ? __ldg(row + idx) : 0.f;
                        }
                    }
#pragma unroll
                    for (int jj = 0; jj < RF; ++jj)
#pragma unroll
                        for (int c = 0; c < NC; ++c) acc[c] = fmaf(aj[jj], v[jj][c], acc[c]);
                }
            }
            const float inv = (w.pool_mean && hi > lo) ? 1.f / (float)(hi - lo) : 1.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int idx = e0 + lane + c * 32;
                if (idx < D) o[idx] = acc[c] * inv;
            }
        }
    }
}

template <bool WT>
static cudaError_t launch_pool_sized(tt_emb* h, int D4, float* out, bool plan, cudaStream_t s)
{
    if (D4 > 8 && D4 <= 16) return launch_pool_async<16, WT>(h, out, plan, s);
    if (D4 > 4 && D4 <= 8) return launch_pool_async<8, WT>(h, out, plan, s);
    if (D4 <= 4) return launch_pool_vec<4, 1, WT>(h, out, plan, s);
    if (D4 <= 32) return launch_pool_vec<32, 1, WT>(h, out, plan, s);
    if (D4 <= 64) return launch_pool_vec<32, 2, WT>(h, out, plan, s);
    if (D4 <= 128) return launch_pool_vec<32, 4, WT>(h, out, plan, s);
    return launch_pool_vec<32, 8, WT>(h, out, plan, s);
}

// rows that k_pool_odd stages (with the up to three floats before a row, its pieces fit the staging row)
#define TT_POOL_ODD_MOST 61
#define TT_POOL_ODD_NARROW 29
template <bool WT>
static cudaError_t launch_pool_unaligned(tt_emb* h, float* out, bool plan, cudaStream_t s)
{
    return h->D <= TT_POOL_ODD_NARROW ? launch_pool_odd<8, WT>(h, out, plan, s) : launch_pool_odd<16, WT>(h, out, plan, s);
}

static bool tt_pool_vectors(const tt_emb* h, const float* out)
{
    return h->D % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
}

cudaError_t tt_plan_pooling(tt_emb* h, const float* out)
{
    h->v.pool_shares = 0;
    if (!tt_pool_vectors(h, out)) {
        if (h->D > TT_POOL_ODD_MOST) return cudaSuccess;   // a warp takes bags, not shares
        return (h->v.psw || h->v.pool_mean) ? launch_pool_unaligned<true>(h, nullptr, true, nullptr) : launch_pool_unaligned<false>(h, nullptr, true, nullptr);
    }
    return (h->v.psw || h->v.pool_mean) ? launch_pool_sized<true>(h, h->D / 4, nullptr, true, nullptr)
                                        : launch_pool_sized<false>(h, h->D / 4, nullptr, true, nullptr);
}

cudaError_t tt_launch_pooling(tt_emb* h, float* out, cudaStream_t s)
{
    WsView& w = h->v;
    const int D = w.D;
    if (!tt_pool_vectors(h, out) && D <= TT_POOL_ODD_MOST)
        return (w.psw || w.pool_mean) ? launch_pool_unaligned<true>(h, out, false, s) : launch_pool_unaligned<false>(h, out, false, s);
    if (!tt_pool_vectors(h, out)) {
        const int64_t want = ((int64_t)w.T * w.B + 7) / 8;  // 8 warps per CTA, one warp per bag
        int pgrid = (int)(want < (int64_t)h->sm_count * 8 ? want : (int64_t)h->sm_count * 8);
        const dim3 pg(pgrid < 1 ? 1 : pgrid);
        cudaError_t e0 = D <= 64 ? tt_launch_pdl(k_pool_scalar<2>, pg, dim3(256), 0, s, w, out)
                       : D <= 128 ? tt_launch_pdl(k_pool_scalar<4>, pg, dim3(256), 0, s, w, out)
                                  : tt_launch_pdl(k_pool_scalar<8>, pg, dim3(256), 0, s, w, out);
        if (e0 != cudaSuccess) return e0;
        tt_note_launch();
        return cudaGetLastError();
    }
    return (w.psw || w.pool_mean) ? launch_pool_sized<true>(h, D / 4, out, false, s) : launch_pool_sized<false>(h, D / 4, out, false, s);
}
