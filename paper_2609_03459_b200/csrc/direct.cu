// Small inference calls: every lookup makes its row for itself and adds it to its bag, in one kernel, without the grouping.
//
// The grouped path is a chain of three to six dependent kernels, most of them grouping, and takes 36 us however little there is to
// do; sharing rows and prefixes pays only where there are many lookups.  Here a warp walks the lookups of a bag (or of its part of one), and
// a row is one chain of products in fp32.  Forward calls, grouped / here, us: 4x4x4: rank 8: 1 k lookups 36.4 / 5.8, 44 k 62 / 27, 107
// k 79 / 53; rank 16: 1 k 39 / 6.4, 7.9 k in 8 tables 61 / 17, 44 k 66 / 43; rank 32: 1 k 48 / 9.1, 16 k 59 / 48; D = 128, rank 32, 1 k 84 / 13; four
// cores, rank 64, 1 k 77 / 41; 3x3x5, 44 k 84 / 61; 8x8, rank 24, 41 k 65 / 34.  Relative error of `out` against 64 bits 1.0e-7 to
// 1.6e-7 (grouped, products of split operands: 1.5e-7 to 4.7e-7).
// Bound by instructions and by latency at sixteen warps per SM (4x4x4, rank 16, 85 k lookups: 436 instructions a lookup, 192 of them
// products and their sums, issue slots 41 to 50 %; 80 registers for 24 warps spill: 90 us instead of 74).
// The inspection calls (grouping_counts, export_level, export_inverse) want the grouping of the last forward: tt_regroup makes it then, from
// the copies of the row ids and offsets that the kernel leaves in the row buffer.
#include "common.cuh"
#include "group.cuh"
#include <type_traits>

#define DIRECT_WARPS 8
#define DIRECT_THREADS (32 * DIRECT_WARPS)
#define DIRECT_MOST_D 128
#define DIRECT_CTAS 2          // 128 registers

__device__ __forceinline__ void direct_cp16(float* smem_dst, const float* gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}

// n contiguous floats into shared memory by one warp; vec: 16-byte aligned, a whole number of float4s
__device__ __forceinline__ void direct_stage(float* dst, const float* __restrict__ src, int n, bool vec, int lane)
{
    if (vec) for (int i = 4 * lane; i < n; i += 128) direct_cp16(dst + i, src + i);
    else for (int i = lane; i < n; i += 32) dst[i] = __ldg(src + i);
}

// row pitch of a partial product in shared memory: rows of whole float4s stay aligned and start in different banks
__host__ __device__ __forceinline__ int direct_pitch(int r) { return (r & 3) == 0 ? r + 4 : (r & 1) == 0 ? r + 2 : r; }

// P_k = P_{k-1} . G_k[i_k] of one lookup by one warp: As M x ra (pitch ap), B ra x cols, result as (M d_k) rows of r (pitch pp).
// A lane owns VW neighbouring columns of MB rows and has four to eight rows of B on their way; `ready` runs once, when the first loads
// are under way.  ra and ap are multiples of four, of r and cols VW is a divisor.
template <int MB, int VW, class Ready>
__device__ __forceinline__ void direct_product(const float* As, int ap, const float* __restrict__ B, int M, int ra, int cols, float* Ps, int r, int pp,
                                               int dk, int lane, Ready& ready)
{
    using Vec = typename std::conditional<VW == 2, float2, float>::type;
    for (int m0 = 0; m0 < M; m0 += MB)
        for (int c0 = 0; c0 < cols; c0 += 32 * VW) {
            const int c = c0 + VW * lane;
            const Vec* __restrict__ Bc = reinterpret_cast<const Vec*>(B + (c < cols ? c : 0));
            const int step = cols / VW;
            Vec b[2][4];
            auto load = [&](Vec (&v)[4]) {
#pragma unroll
                for (int u = 0; u < 4; ++u) { v[u] = __ldg(Bc); Bc += step; }
            };
            load(b[0]);
            if (ra > 4) load(b[1]);
            if (m0 == 0 && c0 == 0) ready();
            float acc[MB][VW];
#pragma unroll
            for (int m = 0; m < MB; ++m)
#pragma unroll
                for (int x = 0; x < VW; ++x) acc[m][x] = 0.f;
            const float* row = As + m0 * ap;
            auto add = [&](const Vec (&v)[4], int a0) {
#pragma unroll
                for (int m = 0; m < MB; ++m) {
                    const float4 a = *reinterpret_cast<const float4*>(row + (m0 + m < M ? m : 0) * ap + a0);
                    const float y[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if constexpr (VW == 2) { acc[m][0] = fmaf(y[u], v[u].x, acc[m][0]); acc[m][VW - 1] = fmaf(y[u], v[u].y, acc[m][VW - 1]); }
                        else acc[m][0] = fmaf(y[u], v[u], acc[m][0]);
                    }
                }
            };
#pragma unroll 1
            for (int a0 = 0; a0 < ra; a0 += 8) {
                add(b[0], a0);
                if (a0 + 8 < ra) load(b[0]);
                if (a0 + 4 >= ra) break;
                add(b[1], a0 + 4);
                if (a0 + 12 < ra) load(b[1]);
            }
            if (c < cols) {
                const int dd = c / r, bb = c - dd * r;
                float* dst = Ps + (m0 * dk + dd) * pp + bb;
#pragma unroll
                for (int m = 0; m < MB; ++m, dst += dk * pp)
                    if (m0 + m < M) {
                        if constexpr (VW == 2) *reinterpret_cast<float2*>(dst) = make_float2(acc[m][0], acc[m][VW - 1]);
                        else *dst = acc[m][0];
                    }
            }
        }
}
// ... of any shape
template <class Ready>
__device__ __forceinline__ void direct_product_any(const float* As, int ap, const float* __restrict__ B, int M, int ra, int cols, float* Ps, int r, int pp,
                                                   int dk, int lane, Ready& ready)
{
    ready();
    for (int m0 = 0; m0 < M; m0 += 4)
        for (int c = lane; c < cols; c += 32) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            const float* row = As + m0 * ap;
#pragma unroll 4
            for (int a = 0; a < ra; ++a) {
                const float x = __ldg(B + a * cols + c);
#pragma unroll
                for (int m = 0; m < 4; ++m) acc[m] = fmaf(row[(m0 + m < M ? m : 0) * ap + a], x, acc[m]);
            }
            const int dd = c / r, bb = c - dd * r;
            float* dst = Ps + (m0 * dk + dd) * pp + bb;
#pragma unroll
            for (int m = 0; m < 4; ++m, dst += dk * pp)
                if (m0 + m < M) *dst = acc[m];
        }
}

template <int KIND, class Ready>
__device__ __forceinline__ void direct_level(const float* As, int ap, const float* __restrict__ B, int M, int ra, int dk, int r, float* Ps, int lane, Ready ready)
{
    const int cols = dk * r, pp = direct_pitch(r);
    if constexpr (KIND == 0) {
        direct_product_any(As, ap, B, M, ra, cols, Ps, r, pp, dk, lane, ready);
    } else {
        constexpr int MB = KIND == 1 ? 4 : 2;
        if (cols > 32) direct_product<MB, 2>(As, ap, B, M, ra, cols, Ps, r, pp, dk, lane, ready);
        else direct_product<MB, 1>(As, ap, B, M, ra, cols, Ps, r, pp, dk, lane, ready);
    }
}

// Lookups `todo` of a chunk (lane i holds the digits and the factor of lookup i), three cores with d_3 = 4: M = d_1, DK = d_2, R = r_2, and
// r_1 a multiple of four up to 32.  The slices of the first and last core of the next lookup are on their way to shared memory while this
// one is multiplied, and so are the first eight rows of its slice of the second core, in registers.  part += row (four columns per
// lane of the first M DK; with few rows of C, its sums over r_2 are cut over groups of lanes: the caller adds them up per bag).
#define DIRECT_SLICE 128      // floats of a staged slice of the first or last core at most
template <int M, int DK, int R> struct DirectShape {
    static constexpr int COLS = DK * R, VW = COLS >= 64 ? 2 : 1, ITEMS = M * DK, CP = R + 4;
    static constexpr int splits(int s) { return 2 * s * ITEMS <= 32 && R / 4 % (2 * s) == 0 ? splits(2 * s) : s; }
    static constexpr int SPLITS = splits(1), LEN = R / SPLITS;
};
template <int M, int DK, int R, bool WT>
__device__ __forceinline__ void direct_chunk(const TableDesc& td, float* sm, unsigned todo, uint32_t i_first, uint32_t i_mid, uint32_t i_last, float wt,
                                             float (&part)[4], int lane)
{
    using S = DirectShape<M, DK, R>;
    constexpr int COLS = S::COLS, VW = S::VW, CP = S::CP;
    using Vec = typename std::conditional<VW == 2, float2, float>::type;
    const int ra = td.r[1], an = M * ra;
    float* const Cs = sm + 4 * DIRECT_SLICE;
    const bool on_a = 4 * lane < an, on_d = 4 * lane < 4 * R, on_b = COLS >= 32 || lane < COLS;
    const float* const gA = td.core[0] + 4 * lane;
    const float* const gD = td.core[2] + 4 * lane;
    const Vec* const gB = reinterpret_cast<const Vec*>(td.core[1]) + (on_b ? lane : 0);
    auto stage = [&](int src, int buf) {
        const uint32_t x = __shfl_sync(0xffffffffu, i_first, src), y = __shfl_sync(0xffffffffu, i_last, src);
        if (on_a) direct_cp16(sm + buf * DIRECT_SLICE + 4 * lane, gA + (size_t)x * (uint32_t)an);
        if (on_d) direct_cp16(sm + (2 + buf) * DIRECT_SLICE + 4 * lane, gD + (size_t)y * (uint32_t)(4 * R));
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    Vec b[2][4];
    auto load = [&](Vec (&v)[4], const Vec* __restrict__ p) {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __ldg(p + u * (COLS / VW));
    };
    const Vec* B = nullptr;
    auto begin = [&](int src) {
        B = gB + (size_t)__shfl_sync(0xffffffffu, i_mid, src) * (uint32_t)(ra * (COLS / VW));
        load(b[0], B);
        if (ra > 4) load(b[1], B + 4 * (COLS / VW));
    };
    int src = __ffs(todo) - 1, buf = 0;
    stage(src, 0);
    begin(src);
    for (;;) {
        todo &= todo - 1;
        const int nsrc = __ffs(todo) - 1;
        const float wj = WT ? __shfl_sync(0xffffffffu, wt, src) : 1.f;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        if (todo) stage(nsrc, buf ^ 1);
        const float* const As = sm + buf * DIRECT_SLICE;
#pragma unroll 1
        for (int c0 = 0; c0 < COLS; c0 += 32 * VW) {
            float acc[M][VW];
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int x = 0; x < VW; ++x) acc[m][x] = 0.f;
            auto add = [&](const Vec (&v)[4], const float* row) {
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const float4 a = *reinterpret_cast<const float4*>(row + m * ra);
                    const float y[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if constexpr (VW == 2) { acc[m][0] = fmaf(y[u], v[u].x, acc[m][0]); acc[m][VW - 1] = fmaf(y[u], v[u].y, acc[m][VW - 1]); }
                        else acc[m][0] = fmaf(y[u], v[u], acc[m][0]);
                    }
                }
            };
            const Vec* p = B + c0 / VW + 8 * (COLS / VW);
#pragma unroll 1
            for (int a0 = 0; a0 < ra; a0 += 8, p += 8 * (COLS / VW)) {
                add(b[0], As + a0);
                if (a0 + 8 < ra) load(b[0], p);
                if (a0 + 4 >= ra) break;
                add(b[1], As + a0 + 4);
                if (a0 + 12 < ra) load(b[1], p + 4 * (COLS / VW));
            }
            if (c0 + 32 * VW < COLS) {     // the next columns
                const Vec* n = B + (c0 + 32 * VW) / VW;
                load(b[0], n);
                if (ra > 4) load(b[1], n + 4 * (COLS / VW));
            }
            const int c = c0 + VW * lane, dd = c / R, bb = c % R;
            if (on_b)
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    float* dst = Cs + (m * DK + dd) * CP + bb;
                    if constexpr (VW == 2) *reinterpret_cast<float2*>(dst) = make_float2(acc[m][0], acc[m][VW - 1]);
                    else *dst = acc[m][0];
                }
        }
        if (todo) begin(nsrc);
        __syncwarp();
        if (lane < S::SPLITS * S::ITEMS) {
            const int item = lane % S::ITEMS, from = lane / S::ITEMS * S::LEN;
            const float* c = Cs + item * CP + from;
            const float4* d = reinterpret_cast<const float4*>(sm + (2 + buf) * DIRECT_SLICE) + from;
            float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int x = 0; x < S::LEN; x += 4) {
                const float4 y = *reinterpret_cast<const float4*>(c + x);
                const float4 e0 = d[x], e1 = d[x + 1], e2 = d[x + 2], e3 = d[x + 3];
                e.x = fmaf(y.x, e0.x, e.x); e.y = fmaf(y.x, e0.y, e.y); e.z = fmaf(y.x, e0.z, e.z); e.w = fmaf(y.x, e0.w, e.w);
                e.x = fmaf(y.y, e1.x, e.x); e.y = fmaf(y.y, e1.y, e.y); e.z = fmaf(y.y, e1.z, e.z); e.w = fmaf(y.y, e1.w, e.w);
                e.x = fmaf(y.z, e2.x, e.x); e.y = fmaf(y.z, e2.y, e.y); e.z = fmaf(y.z, e2.z, e.z); e.w = fmaf(y.z, e2.w, e.w);
                e.x = fmaf(y.w, e3.x, e.x); e.y = fmaf(y.w, e3.y, e.y); e.z = fmaf(y.w, e3.z, e.z); e.w = fmaf(y.w, e3.w, e.w);
            }
            if (WT) {
                part[0] = fmaf(wj, e.x, part[0]); part[1] = fmaf(wj, e.y, part[1]);
                part[2] = fmaf(wj, e.z, part[2]); part[3] = fmaf(wj, e.w, part[3]);
            } else { part[0] += e.x; part[1] += e.y; part[2] += e.z; part[3] += e.w; }
        }
        if (!todo) break;
        src = nsrc;
        buf ^= 1;
    }
    __syncwarp();
}
// the shape's splits, for the caller
__device__ __forceinline__ int direct_splits(int fast)
{
    switch (fast) {
        case 0: return DirectShape<4, 4, 32>::SPLITS;
        case 1: return DirectShape<4, 4, 16>::SPLITS;
        case 2: return DirectShape<4, 4, 8>::SPLITS;
        case 3: return DirectShape<4, 8, 32>::SPLITS;
        case 5: return DirectShape<2, 4, 32>::SPLITS;
        case 6: return DirectShape<2, 4, 16>::SPLITS;
        case 7: return DirectShape<2, 4, 8>::SPLITS;
        case 8: return DirectShape<2, 2, 32>::SPLITS;
        case 9: return DirectShape<2, 2, 16>::SPLITS;
        default: return DirectShape<2, 2, 8>::SPLITS;
    }
}

// a, p, c, d: floats of shared memory per warp for the slice of the first core, P_2 of four cores, C, the slice of the last core (KIND 3: a
// and p are the two buffers of direct_chunk); 1 << team_log warps make a bag
struct DirectPlan {
    int a, p, c, d, team_log, kind;
};

// KIND: 0 any shape; 1, 2: ranks and d_K multiples of four, 2: P_{K-2} of at most two rows; 3: direct_chunk's shapes.
// A bag's warps take its lookups in turn; their sums meet in shared memory, in order.  The bags after the first of every team are handed
// out through a counter.  Offsets and row ids are checked on the way.  ids, offsets: copies for tt_regroup, in the row buffer, which
// this call does not use.
template <int KIND, bool WT>
__global__ void __launch_bounds__(DIRECT_THREADS, DIRECT_CTAS) k_direct(const __grid_constant__ WsView w, float* __restrict__ out, DirectPlan plan, void* ids, int64_t* offsets)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(16) float s_sum[2][DIRECT_WARPS][DIRECT_MOST_D];   // two bags in turn: one barrier per bag
    __shared__ uint32_t s_next[2][DIRECT_WARPS];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, K = KIND == 3 ? 3 : w.K, D = w.D;
    float* const As = sm + (size_t)wid * (plan.a + plan.p + plan.c + plan.d);
    float *const Ps = As + plan.a, *const Cs = Ps + plan.p, *const Ds = Cs + plan.c;
    const uint32_t W = 1u << plan.team_log, part_of = wid & (W - 1), B = (uint32_t)w.B, nb = (uint32_t)(w.T * w.B), L = (uint32_t)w.L;
    const uint32_t per = DIRECT_WARPS >> plan.team_log;
    auto clampL = [&](int64_t x) { return x < 0 ? 0u : (x > w.L ? L : (uint32_t)x); };
    bool bad_id = false, bad_offset = false;
    uint32_t* const ctr = w.counters + CTR_DIRECT;
    const uint32_t team = wid >> plan.team_log, teams = gridDim.x * per;
    int turn = 0;
    for (uint32_t bag = blockIdx.x * per + team; bag < nb; turn ^= 1) {
        // bags past the first of every team are handed out: their lengths differ
        uint32_t next = nb;
        if (nb > teams && part_of == 0 && lane == 0) next = teams + atomicAdd(ctr + 6, 1u);
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
        const int64_t o = __ldg(w.offsets + bag), o_next = __ldg(w.offsets + bag + 1);
        bad_offset = bad_offset || o < 0 || o > w.L || o_next < o || (bag == 0 && o != 0) || (bag + 1 == nb && o_next != w.L);
        if (part_of == 0 && lane < 2 && (lane == 0 || bag + 1 == nb)) offsets[bag + lane] = lane == 0 ? o : o_next;
        const uint32_t lo = clampL(o), hi = clampL(o_next), t = bag / B, b = bag - t * B;
        const TableDesc& td = w.tdesc[t];
        const int d1 = td.d[0], r1 = td.r[1], an = d1 * r1, dK = td.d[K - 1], rK = td.r[K - 1], dn = rK * dK;
        const int cp = K == 2 ? r1 : direct_pitch(rK);
        const float* const C = K == 2 ? As : Cs;
        const bool avec = KIND > 0 || (an & 3) == 0, dvec = KIND > 0 || (dn & 3) == 0;
        // E = C . G_K[i_K]: an item is four columns of one row of C, the sum over r_{K-1} cut into `splits` where there are few items;
        // shapes that are no multiples of four: one element of E
        const bool quads = KIND > 0 || ((dK & 3) == 0 && (rK & 3) == 0);
        const int items = quads ? D / 4 : D;
        int splits = 1;
        if (KIND == 3) splits = direct_splits(td.fast);
        else if (quads && (items & (items - 1)) == 0)
            while (2 * splits * items <= 32 && ((rK >> 2) & (2 * splits - 1)) == 0) splits *= 2;
        const int q4 = dK >> 2, len = rK / splits;
        const bool on = lane < splits * items;
        const float* e_c = C;
        const float4* e_d = reinterpret_cast<const float4*>(Ds);
        if (quads && on) {
            const int item = lane % items, s = lane / items, p = item / q4;
            e_c += p * cp + s * len;
            e_d += s * len * q4 + item - p * q4;
        }
        for (uint32_t l0 = lo; l0 < hi; l0 += 32 * W) {
            const uint32_t l = l0 + part_of + W * lane;
            uint32_t q = 0;
            bool ok = false;
            float wt = 1.f;
            if (l < hi) {
                const int64_t id = tt_index<true>(w, l);
                if (w.idx32) reinterpret_cast<int32_t*>(ids)[l] = (int32_t)id; else reinterpret_cast<int64_t*>(ids)[l] = id;
                ok = id >= 0 && id < td.N;
                bad_id = bad_id || !ok;
                if (ok) q = (uint32_t)id;
                if (WT && w.psw) wt = __ldg(w.psw + l);
            }
            // digits of this lane's row id
            const uint32_t nK = (uint32_t)td.n[K - 1], i_last = q % nK;
            uint32_t i_mid = 0, i_mid1 = 0;
            q /= nK;
            if (K >= 3) { const uint32_t n = (uint32_t)td.n[K - 2]; i_mid = q % n; q /= n; }
            if (K >= 4) { const uint32_t n = (uint32_t)td.n[1]; i_mid1 = q % n; q /= n; }
            unsigned todo = __ballot_sync(0xffffffffu, ok);
            float part[4] = {0.f, 0.f, 0.f, 0.f};     // two-level sum, as in the pooling kernels
            if constexpr (KIND == 3) {
                if (todo) switch (td.fast) {
                    case 0: direct_chunk<4, 4, 32, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 1: direct_chunk<4, 4, 16, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 2: direct_chunk<4, 4, 8, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 3: direct_chunk<4, 8, 32, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 5: direct_chunk<2, 4, 32, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 6: direct_chunk<2, 4, 16, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 7: direct_chunk<2, 4, 8, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 8: direct_chunk<2, 2, 32, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    case 9: direct_chunk<2, 2, 16, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                    default: direct_chunk<2, 2, 8, WT>(td, As, todo, q, i_mid, i_last, wt, part, lane); break;
                }
            } else {
            while (todo) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1;
                const uint32_t x1 = __shfl_sync(0xffffffffu, q, src), xK = __shfl_sync(0xffffffffu, i_last, src), xm = __shfl_sync(0xffffffffu, i_mid, src);
                const float wj = WT ? __shfl_sync(0xffffffffu, wt, src) : 1.f;
                __syncwarp();                          // the lookup before is done with the shared memory
                direct_stage(As, td.core[0] + (size_t)x1 * an, an, avec, lane);
                direct_stage(Ds, td.core[K - 1] + (size_t)xK * dn, dn, dvec, lane);
                auto staged = [&]() {
                    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                };
                if (K == 2) staged();
                const uint32_t xm1 = K == 4 ? __shfl_sync(0xffffffffu, i_mid1, src) : 0u;
                const float* in = As;
                int M = d1, ra = r1, ap = r1;
#pragma unroll 1
                for (int k = 1; k < K - 1; ++k) {
                    const bool top = k == K - 2;
                    float* to = top ? Cs : Ps;
                    direct_level<KIND>(in, ap, td.core[k] + (size_t)(top ? xm : xm1) * td.slice_floats[k], M, ra, td.d[k], td.r[k + 1], to, lane, staged);
                    in = to;
                    M *= td.d[k];
                    ra = td.r[k + 1];
                    ap = direct_pitch(ra);
                }
                __syncwarp();
                if (quads) {
                    if (on) {
                        float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
                        for (int x = 0; x < len; x += 4) {
                            const float4 y = *reinterpret_cast<const float4*>(e_c + x);
                            const float4 e0 = e_d[x * q4], e1 = e_d[(x + 1) * q4], e2 = e_d[(x + 2) * q4], e3 = e_d[(x + 3) * q4];
                            e.x = fmaf(y.x, e0.x, e.x); e.y = fmaf(y.x, e0.y, e.y); e.z = fmaf(y.x, e0.z, e.z); e.w = fmaf(y.x, e0.w, e.w);
                            e.x = fmaf(y.y, e1.x, e.x); e.y = fmaf(y.y, e1.y, e.y); e.z = fmaf(y.y, e1.z, e.z); e.w = fmaf(y.y, e1.w, e.w);
                            e.x = fmaf(y.z, e2.x, e.x); e.y = fmaf(y.z, e2.y, e.y); e.z = fmaf(y.z, e2.z, e.z); e.w = fmaf(y.z, e2.w, e.w);
                            e.x = fmaf(y.w, e3.x, e.x); e.y = fmaf(y.w, e3.y, e.y); e.z = fmaf(y.w, e3.z, e.z); e.w = fmaf(y.w, e3.w, e.w);
                        }
                        part[0] = fmaf(wj, e.x, part[0]); part[1] = fmaf(wj, e.y, part[1]);
                        part[2] = fmaf(wj, e.z, part[2]); part[3] = fmaf(wj, e.w, part[3]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int e = lane + 32 * i;
                        if (e >= D) break;
                        const int p = e / dK, j = e - p * dK;
                        float x = 0.f;
#pragma unroll 4
                        for (int a = 0; a < rK; ++a) x = fmaf(C[p * cp + a], Ds[a * dK + j], x);
                        part[i] = fmaf(wj, x, part[i]);
                    }
                }
            }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[i] += part[i];
        }
        // the pieces of the sums over r_{K-1} meet once per bag
        if (quads)
            for (int o = items; o < splits * items; o <<= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
        if (W > 1) {    // the warps of the bag, in order
            float (*const sums)[DIRECT_MOST_D] = s_sum[turn] + wid;
            if (part_of > 0) {
                if (quads) {
                    if (lane < items) *reinterpret_cast<float4*>(&sums[0][4 * lane]) = make_float4(sum[0], sum[1], sum[2], sum[3]);
                } else
#pragma unroll
                    for (int i = 0; i < 4; ++i) sums[0][lane + 32 * i] = sum[i];
            } else if (lane == 0) s_next[turn][team] = next;
            asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(32 * W) : "memory");
            next = s_next[turn][team];
            if (part_of == 0)
                for (uint32_t x = 1; x < W; ++x)
#pragma unroll
                    for (int i = 0; i < 4; ++i) sum[i] += sums[x][quads ? 4 * lane + i : lane + 32 * i];
        } else next = __shfl_sync(0xffffffffu, next, 0);
        if (part_of == 0) {
            if (WT && w.pool_mean && hi > lo) {
                const float inv = 1.f / (float)(hi - lo);
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[i] *= inv;
            }
            float* o = out + ((size_t)b * w.T + t) * D;
            if (quads) {
                if (lane < items) {
                    if ((reinterpret_cast<uintptr_t>(out) & 15) == 0) __stcs(reinterpret_cast<float4*>(o) + lane, make_float4(sum[0], sum[1], sum[2], sum[3]));
                    else
#pragma unroll
                        for (int i = 0; i < 4; ++i) o[4 * lane + i] = sum[i];
                }
            } else
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (lane + 32 * i < D) __stcs(o + lane + 32 * i, sum[i]);
        }
        bag = next;
    }
    // the status word is written by the CTA that reports last (nobody waits), which leaves the counters of this kernel at zero
    const int bits = (__syncthreads_or(bad_id) ? TT_EMB_STATUS_INDEX : 0) | (__syncthreads_or(bad_offset) ? TT_EMB_STATUS_OFFSETS : 0);
    if (threadIdx.x == 0) {
        if (bits) atomicOr(ctr + 1, (uint32_t)bits);
        __threadfence();
        s_last = atomicAdd(ctr, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    uint32_t all = __ldcg(ctr + 1);
    if (all & TT_EMB_STATUS_OFFSETS) {   // the bags need not cover the lookups, nor each lookup be in a bag of its table
        bool bad = false;
        for (uint32_t l = threadIdx.x; l < L; l += DIRECT_THREADS) {
            int t = 0, hi = w.T;
            while (hi - t > 1) {
                const int mid = (t + hi) >> 1;
                if (tt_table_start(w, mid) <= l) t = mid; else hi = mid;
            }
            const int64_t id = tt_index(w, l);
            if (w.idx32) reinterpret_cast<int32_t*>(ids)[l] = (int32_t)id; else reinterpret_cast<int64_t*>(ids)[l] = id;
            bad = bad || id < 0 || id >= w.tdesc[t].N;
        }
        all = TT_EMB_STATUS_OFFSETS | (__syncthreads_or(bad) ? TT_EMB_STATUS_INDEX : 0);
    }
    if (threadIdx.x == 0) {
        *w.status = (int32_t)all;
        ctr[0] = 0u;
        ctr[1] = 0u;
        ctr[2] = 1u;           // not grouped: tt_regroup
        ctr[3] = B;
        ctr[4] = L;
        ctr[5] = (uint32_t)w.idx32;
        ctr[6] = 0u;
    }
}

// The row buffer holds the copies of the offsets, then of the row ids
static size_t direct_copy_bytes(const tt_emb* h) { return ((size_t)h->T * h->v.B + 1 + (size_t)h->v.L) * sizeof(int64_t); }

#define DIRECT_MOST_SMEM (100 << 10)
#define DIRECT_FEWEST_BAGS 64          // with fewer, one long bag keeps the call waiting
#define DIRECT_MOST_LOOKUPS (1 << 18)
// Whether the call is made this way, and how: the time that it would take against that of the grouped path, both as fitted to forward
// calls of eleven shapes, 1 to 16 tables, 64 to 65536 bags each, 1 k to 0.2 M lookups (us).
//   here      a lookup takes the chip 0.3 ns and its products or slices, whichever is longer (4x4x4, rank 8 / 16 / 32: 0.47 / 0.83 / 2.6
//             ns; D = 128 4.8; four cores, rank 64 25), a bag 0.28 ns; and a warp makes its lookups one after the other (one table, 64 bags of 55
//             lookups, eight warps each, rank 16 / 32 / 64: 17 / 48 / 445 us), a bag of 1.6 times the average length among them.
//   grouped   36 to 84 us with 1 k lookups, by shape, and 0.28 ns for each of the others.
// Near the line both take the same (4x4x4, rank 16: 107 k lookups 87 / 90; rank 8: 203 k 100 / 92; 2x2x4, rank 32: 107 k 102 / 105).
// Warps of a bag: its lookups by eight, or by two where the bags are few.  With 1 / 2 / 4 / 8 warps, rank 16: bags of 1 lookup, 16 k
// of them 26 / 42 / 78 / 152; of 1 to 20, 768 of them 24 / 17 / 18 / 17, 4096 51 / 43 / 45 / 59; of 1 to 100, 64 of them 92 / 48 / 26 / 17, 4096
// 217 / 165 / 147 / 155.
static bool direct_plan(const tt_emb* h, DirectPlan& plan)
{
    const WsView& w = h->v;
    const int K = h->K;
    plan = DirectPlan{};
    if (h->enable_backward || h->ablation || h->D > DIRECT_MOST_D) return false;
    const int64_t nb = (int64_t)h->T * w.B;
    if (nb < DIRECT_FEWEST_BAGS || w.L > DIRECT_MOST_LOOKUPS || direct_copy_bytes(h) > (size_t)h->capU * h->D * sizeof(float)) return false;
    int64_t rows = 0;
    double products = 0, bytes = 0;      // per lookup
    bool fast = true;
    plan.kind = 2;
    for (int t = 0; t < h->T; ++t) {
        const TableDesc& td = h->tab[t];
        rows += td.N;
        bool fours = (td.d[K - 1] & 3) == 0;
        for (int k = 1; k < K; ++k) {
            fours = fours && (td.r[k] & 3) == 0;
            products += (double)td.P[k] * td.slice_floats[k];
            bytes += 4.0 * td.slice_floats[k];
        }
        if (!fours) plan.kind = 0;
        else if (plan.kind == 2 && td.P[K - 2] > 2) plan.kind = 1;
        auto most = [](int& x, int y) { y = (y + 3) & ~3; if (y > x) x = y; };
        most(plan.a, td.d[0] * td.r[1]);
        if (K != 3 || td.fast < 0 || td.fast == 4 || (td.r[1] & 3) || td.d[0] * td.r[1] > DIRECT_SLICE) fast = false;
        if (K == 4) most(plan.p, td.P[2] * direct_pitch(td.r[2]));
        if (K >= 3) most(plan.c, td.P[K - 1] * direct_pitch(td.r[K - 1]));
        most(plan.d, td.slice_floats[K - 1]);
    }
    if (fast) {
        plan.kind = 3;
        plan.a = plan.p = 2 * DIRECT_SLICE;
        plan.d = 0;
    }
    // with a row buffer for fewer rows the surplus is dropped, and which rows these are shows in the grouping
    if (h->capU < w.L && h->capU < rows) return false;
    if ((plan.a + plan.p + plan.c + plan.d) * DIRECT_WARPS * sizeof(float) > DIRECT_MOST_SMEM) return false;
    // warps of a bag
    products /= h->T;
    bytes /= h->T;
    const double bag = (double)w.L / (double)nb;
    int W = 1;
    while (W < DIRECT_WARPS && (bag >= 8 * W || (bag >= 2 * W && nb * W <= (int64_t)h->sm_count * 4))) { W *= 2; ++plan.team_log; }
    const double lookups = (double)w.L * (0.3e-3 + (products > bytes / 1.5 ? products : bytes / 1.5) / 8.5e6 + (fast ? 0 : 0.5e-3)) + (double)nb * 0.28e-3;
    const double chain = bag <= 1 ? 0 : 1.6 * bag / W * (0.6 + products / 5000);
    const double grouped = 38 + 0.28e-3 * (double)w.L + (products < 45000 ? products / 1500 : 30);
    return lookups <= grouped && chain <= grouped;
}

// launched: whether the call is made this way
cudaError_t tt_launch_direct(tt_emb* h, float* out, bool* launched, cudaStream_t s)
{
    const WsView& w = h->v;
    DirectPlan plan;
    *launched = false;
    if (!direct_plan(h, plan)) return cudaSuccess;
    *launched = true;
    const size_t smem = (size_t)(plan.a + plan.p + plan.c + plan.d) * DIRECT_WARPS * sizeof(float);
    const bool wt = w.psw || w.pool_mean;
    auto kern = plan.kind == 3 ? (wt ? k_direct<3, true> : k_direct<3, false>) : plan.kind == 0 ? (wt ? k_direct<0, true> : k_direct<0, false>)
              : plan.kind == 1 ? (wt ? k_direct<1, true> : k_direct<1, false>) : (wt ? k_direct<2, true> : k_direct<2, false>);
    cudaError_t e;
    int& per_sm = h->direct_ctas[wt];     // kernel and shared memory are those of the handle's tables: asked once
    if (per_sm == 0) {
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, DIRECT_MOST_SMEM)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, DIRECT_THREADS, smem)) != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
    }
    const int64_t need = ((((int64_t)h->T * w.B) << plan.team_log) + DIRECT_WARPS - 1) / DIRECT_WARPS, most = (int64_t)h->sm_count * per_sm;
    int64_t* offsets = reinterpret_cast<int64_t*>(w.E);
    if ((e = tt_launch_pdl(kern, dim3((unsigned)(need < most ? need : most)), dim3(DIRECT_THREADS), smem, s, w, out, plan, (void*)(offsets + (size_t)h->T * w.B + 1), offsets)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

cudaError_t tt_regroup(tt_emb* h, cudaStream_t s)
{
    WsView& w = h->v;
    uint32_t say[4];
    cudaError_t e = cudaMemcpyAsync(say, w.counters + CTR_DIRECT + 2, sizeof(say), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess || (e = cudaStreamSynchronize(s)) != cudaSuccess || say[0] == 0u) return e;
    const WsView before = w;
    w.B = say[1];
    w.L = say[2];
    w.idx32 = (int32_t)say[3];
    w.offsets = reinterpret_cast<const int64_t*>(w.E);
    w.indices = w.offsets + (size_t)h->T * w.B + 1;
    w.pool_shares = 0;
    e = tt_launch_grouping(h, s);
    if (e == cudaSuccess) e = tt_launch_schedule(h, s);
    w = before;
    return e;
}
