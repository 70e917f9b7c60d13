// Batches of groups for the sweeps of shapes without a register-tiled variant (any K, dim factors and ranks).
//
// A CTA takes up to GEN_GROUPS groups of its work unit at a time, as many as their C tiles (P_{K-1} x r_{K-1} each) fit in
// shared memory, and spreads every step flat over its threads: the products C = P . G_{K-1}[i] over (group, column), the
// rows over (row, rows of C, columns).  One group at a time (the former shape of these kernels) left most threads idle:
// a group of 3x3x5 has 12 columns and 8 rows, and paid five barriers and a chain of dependent look-ups.  Bound by the
// operand loads (one shared-memory or L1 load for two to four products; the shapes are arbitrary, so nothing is unrolled to
// register tiles).  3x3x5, ranks 6 and 4, 1 M lookups: forward sweep 215 -> 65 us, backward 332 -> 163 us; 8x8, rank 24, K = 2,
// 24 k lookups in 4 tables: the training call 1.43 -> 0.20 ms (few groups of up to 2000 rows each: units are ranges of rows).
#pragma once
#include "common.cuh"

#define GEN_THREADS 256
#define GEN_GROUPS 32
#define GEN_ROWS 256        // rows whose addresses are looked up at a time
#define GEN_C_FLOATS 8192   // shared memory for C tiles; one tile has at most 4096 floats and its padding at most 1024

struct GenBatch {
    uint32_t g[GEN_GROUPS], val[GEN_GROUPS], u0[GEN_GROUPS];
    uint32_t row0[GEN_GROUPS + 1];        // rows of the batch before this group
    uint32_t part[GEN_GROUPS];            // some of the group's rows belong to another unit
    const float* left[GEN_GROUPS];        // P_{K-2} of the group (K = 2: its C)
    uint32_t u[GEN_ROWS];                 // rows of the current chunk: slot, group of the batch, slice of the last core
    uint32_t q[GEN_ROWS];
    uint32_t iK[GEN_ROWS];
};

// row pitch of C in shared memory: odd, so that neighbouring rows of C lie in different banks
__host__ __device__ __forceinline__ int gen_pitch(int rb) { return rb | 1; }

// groups [g0, g1) of a work unit and the range of its rows.  K >= 3: whole groups.  K = 2 has few groups with up to n_2 rows
// each, so its units are ranges of rows (the rows of neighbouring groups are neighbours) and may start and end inside a
// group.  Called by all threads, no barrier.
__device__ __forceinline__ void gen_unit(const WsView& w, int t, uint2 rng, uint2& groups, uint2& rows)
{
    if (w.K >= 3) {
        groups = rng;
        rows = make_uint2(0u, 0xffffffffu);
        return;
    }
    rows = rng;
    groups = make_uint2(0u, 0u);
    if (rng.x >= rng.y) return;
    auto holder = [&](uint32_t u) {      // the group of row u
        uint32_t lo = w.tb[1][t], hi = w.tb[1][t + 1];
        while (hi - lo > 1) {
            const uint32_t mid = lo + ((hi - lo) >> 1);
            if (w.cstart[1][mid] <= u) lo = mid; else hi = mid;
        }
        return lo;
    };
    groups = make_uint2(holder(rng.x), holder(rng.y - 1) + 1);
}

// look up groups base .. base + cnt of the unit (ends with a barrier)
__device__ __forceinline__ void gen_batch_begin(const WsView& w, const TableDesc& td, uint32_t base, int cnt, uint2 rows, GenBatch& b)
{
    const int K = w.K;
    if (threadIdx.x < 32) {
        const int i = threadIdx.x;
        uint32_t n = 0;
        if (i < cnt) {
            const uint32_t pos = base + i;
            const uint32_t g = tt_digit_major(w) ? w.tnode[K - 1][pos] : pos;
            b.g[i] = g;
            b.val[i] = w.val[K - 1][g];
            const uint32_t u0 = w.cstart[K - 1][g], u1 = w.cstart[K - 1][g + 1];
            b.u0[i] = max(u0, rows.x);
            n = min(u1, rows.y) - b.u0[i];
            b.part[i] = n != u1 - u0;
            b.left[i] = K >= 3 ? tt_left_operand(w, td, K - 1, g) : td.core[0] + (size_t)b.val[i] * td.slice_floats[0];
        }
        uint32_t incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (i >= o) incl += y;
        }
        b.row0[i + 1] = incl;
        if (i == 0) b.row0[0] = 0;
    }
    __syncthreads();
}

// C of every group of the batch into Cs (ends with a barrier)
__device__ __forceinline__ void gen_batch_c(const WsView& w, const TableDesc& td, int cnt, const GenBatch& b, float* Cs)
{
    const int K = w.K, km = K - 2, Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb), tile = Pm * pitch;
    if (K >= 3) {
        constexpr int MB = 8;
        const int M = td.P[km], ra = td.r[km], dm = td.d[km], cols = dm * rb, mblocks = (M + MB - 1) / MB;
        for (int it = threadIdx.x; it < cnt * mblocks * cols; it += GEN_THREADS) {
            const int c = it % cols, qm = it / cols, q = qm / mblocks, m0 = (qm - q * mblocks) * MB, mm = min(MB, M - m0);
            const float* P = b.left[q] + m0 * ra;
            const float* B = td.core[km] + (size_t)(b.val[q] % (uint32_t)td.n[km]) * td.slice_floats[km] + c;
            float acc[MB];
#pragma unroll
            for (int i = 0; i < MB; ++i) acc[i] = 0.f;
#pragma unroll 4
            for (int a = 0; a < ra; ++a) {
                const float x = __ldg(B + (size_t)a * cols);
#pragma unroll
                for (int i = 0; i < MB; ++i) acc[i] = fmaf(i < mm ? P[i * ra + a] : 0.f, x, acc[i]);
            }
            const int j = c / rb;
            float* dst = Cs + q * tile + (m0 * dm + j) * pitch + (c - j * rb);
#pragma unroll
            for (int i = 0; i < MB; ++i)
                if (i < mm) dst[i * dm * pitch] = acc[i];
        }
    } else {
        for (int it = threadIdx.x; it < cnt * Pm * rb; it += GEN_THREADS) {
            const int q = it / (Pm * rb), e = it - q * (Pm * rb), p = e / rb;
            Cs[q * tile + p * pitch + (e - p * rb)] = b.left[q][e];
        }
    }
    __syncthreads();
}

// look up rows r0 .. r0 + n of the batch (ends with a barrier)
__device__ __forceinline__ void gen_rows(const WsView& w, const TableDesc& td, int cnt, uint32_t r0, int n, GenBatch& b)
{
    static_assert(GEN_ROWS == GEN_THREADS, "one row per thread");
    if ((int)threadIdx.x < n) {
        const uint32_t r = r0 + threadIdx.x;
        int lo = 0, hi = cnt;             // the group that holds row r
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (b.row0[mid] <= r) lo = mid; else hi = mid;
        }
        const uint32_t u = b.u0[lo] + (r - b.row0[lo]);
        b.u[threadIdx.x] = u;
        b.q[threadIdx.x] = (uint32_t)lo;
        b.iK[threadIdx.x] = w.val[w.K][u] - b.val[lo] * (uint32_t)td.n[w.K - 1];
    }
    __syncthreads();
}

// groups per batch of a table
__device__ __forceinline__ int gen_groups(const TableDesc& td, int K)
{
    const int tile = td.P[K - 1] * gen_pitch(td.r[K - 1]);
    return min(GEN_GROUPS, GEN_C_FLOATS / tile);
}

// x[0..3] = the four floats at p, of which `n` exist; VEC: p is 16-byte aligned and n = 4
template <bool VEC>
__device__ __forceinline__ void gen_load4(float (&x)[4], const float* __restrict__ p, int n)
{
    if (VEC) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = i < n ? __ldg(p + i) : 0.f;
    }
}

__device__ __forceinline__ void gen_red4(float* p, const float (&x)[4])
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]) : "memory");
}

// E = C . G_K[i_K] of the n looked-up rows: an item is two rows of C by four columns of the slice
template <bool VEC>
__device__ __forceinline__ void gen_forward_rows(const WsView& w, const TableDesc& td, int n, const GenBatch& b, const float* Cs)
{
    const int K = w.K, Pm = td.P[K - 1], rb = td.r[K - 1], dK = td.d[K - 1], pitch = gen_pitch(rb);
    const int jb = (dK + 3) / 4, pb = (Pm + 1) / 2, per = pb * jb;
    for (int it = threadIdx.x; it < n * per; it += GEN_THREADS) {
        const int i = it / per, e = it - i * per, p = e / jb * 2, j = (e - e / jb * jb) * 4;
        const int nj = min(4, dK - j);
        const float* c0 = Cs + b.q[i] * (Pm * pitch) + p * pitch;
        const float* c1 = p + 1 < Pm ? c0 + pitch : c0;
        const float* D = td.core[K - 1] + (size_t)b.iK[i] * td.slice_floats[K - 1] + j;
        float x0[4] = {0.f, 0.f, 0.f, 0.f}, x1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int a = 0; a < rb; ++a) {
            float d[4];
            gen_load4<VEC>(d, D + a * dK, nj);
            const float y0 = c0[a], y1 = c1[a];
#pragma unroll
            for (int x = 0; x < 4; ++x) { x0[x] = fmaf(y0, d[x], x0[x]); x1[x] = fmaf(y1, d[x], x1[x]); }
        }
        float* o = w.E + (size_t)b.u[i] * w.D + p * dK + j;
        if (VEC) {
            *reinterpret_cast<float4*>(o) = make_float4(x0[0], x0[1], x0[2], x0[3]);
            if (p + 1 < Pm) *reinterpret_cast<float4*>(o + dK) = make_float4(x1[0], x1[1], x1[2], x1[3]);
        } else {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if (x < nj) o[x] = x0[x];
                if (x < nj && p + 1 < Pm) o[dK + x] = x1[x];
            }
        }
    }
}

// dG_K[i_K] += C^T . dE of the n looked-up rows, added to the table's partial copy `gk` with reductions.  VEC: an item is two
// rows of the slice by four columns (one load of dE feeds eight products), otherwise four neighbouring elements
template <bool VEC>
__device__ __forceinline__ void gen_backward_slice(const WsView& w, const TableDesc& td, int n, const GenBatch& b, const float* Cs, float* gk)
{
    const int K = w.K, Pm = td.P[K - 1], rb = td.r[K - 1], dK = td.d[K - 1], pitch = gen_pitch(rb), slice = td.slice_floats[K - 1];
    const int jb = dK / 4, per = VEC ? (rb + 1) / 2 * jb : (slice + 3) / 4;
    for (int it = threadIdx.x; it < n * per; it += GEN_THREADS) {
        const int i = it / per, e = it - i * per;
        const float* c = Cs + b.q[i] * (Pm * pitch);
        const float* dE = w.E + (size_t)b.u[i] * w.D;
        float* dst = gk + (size_t)b.iK[i] * slice;
        if (VEC) {
            const int a = e / jb * 2, j = (e - e / jb * jb) * 4;
            const bool two = a + 1 < rb;
            const float* ca = c + a;
            float x0[4] = {0.f, 0.f, 0.f, 0.f}, x1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int p = 0; p < Pm; ++p) {
                const float4 d = *reinterpret_cast<const float4*>(dE + p * dK + j);
                const float y0 = ca[p * pitch], y1 = two ? ca[p * pitch + 1] : 0.f;
                x0[0] = fmaf(y0, d.x, x0[0]); x0[1] = fmaf(y0, d.y, x0[1]); x0[2] = fmaf(y0, d.z, x0[2]); x0[3] = fmaf(y0, d.w, x0[3]);
                x1[0] = fmaf(y1, d.x, x1[0]); x1[1] = fmaf(y1, d.y, x1[1]); x1[2] = fmaf(y1, d.z, x1[2]); x1[3] = fmaf(y1, d.w, x1[3]);
            }
            gen_red4(dst + a * dK + j, x0);
            if (two) gen_red4(dst + (a + 1) * dK + j, x1);
        } else {
            int pa[4], pj[4];
            float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 4; ++k) { const int s = min(4 * e + k, slice - 1); pa[k] = s / dK; pj[k] = s - pa[k] * dK; }
#pragma unroll 2
            for (int p = 0; p < Pm; ++p)
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] = fmaf(c[p * pitch + pa[k]], dE[p * dK + pj[k]], x[k]);
            if ((slice & 3) == 0) gen_red4(dst + 4 * e, x);
            else
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (4 * e + k < slice) atomicAdd(dst + 4 * e + k, x[k]);
        }
    }
}

// dC += dE . G_K[i_K]^T over the n looked-up rows, r0 the first of them: an item is two by two elements of one group's dC
// over the group's rows among them, eight rows to a partial sum.  Where the rows belong to few groups, a group's rows are
// cut into `parts` so that all threads have an item; the parts meet in s_part [GEN_THREADS] and are added in order.
template <bool VEC>
__device__ __forceinline__ void gen_backward_dc(const WsView& w, const TableDesc& td, uint32_t r0, int n, const GenBatch& b, float* dCs, float4* s_part)
{
    const int K = w.K, Pm = td.P[K - 1], rb = td.r[K - 1], dK = td.d[K - 1], pitch = gen_pitch(rb), slice = td.slice_floats[K - 1];
    const int q0 = (int)b.q[0], nq = (int)b.q[n - 1] - q0 + 1, ab = (rb + 1) / 2, per = (Pm + 1) / 2 * ab, items = nq * per;
    const int parts = items < GEN_THREADS ? min(16, GEN_THREADS / items) : 1;
    auto add = [&](int ie, const float4& x) {
        const int qq = ie / per, e = ie - qq * per, p = e / ab * 2, a = (e - e / ab * ab) * 2;
        float* dst = dCs + (q0 + qq) * (Pm * pitch) + p * pitch + a;
        dst[0] += x.x;
        if (a + 1 < rb) dst[1] += x.y;
        if (p + 1 < Pm) dst[pitch] += x.z;
        if (p + 1 < Pm && a + 1 < rb) dst[pitch + 1] += x.w;
    };
    for (int it = threadIdx.x; it < items * parts; it += GEN_THREADS) {
        const int part = it / items, ie = it - part * items, qq = ie / per, e = ie - qq * per, p = e / ab * 2, a = (e - e / ab * ab) * 2;
        const int q = q0 + qq;
        int i0 = b.row0[q] > r0 ? (int)(b.row0[q] - r0) : 0, i1 = min(n, (int)(b.row0[q + 1] - r0));
        const int len = (i1 - i0 + parts - 1) / parts;
        i0 += part * len;
        i1 = min(i1, i0 + len);
        const int pn = p + 1 < Pm ? dK : 0, an = a + 1 < rb ? dK : 0;   // to the second row of dE, of the slice (none: the first again)
        float sum[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
        for (int ib = i0; ib < i1; ib += 8) {
            float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
            const int ie8 = min(i1, ib + 8);
#pragma unroll 2
            for (int i = ib; i < ie8; ++i) {
                const float* D = td.core[K - 1] + (size_t)b.iK[i] * slice + a * dK;
                const float* dE = w.E + (size_t)b.u[i] * w.D + p * dK;
                for (int j = 0; j < dK; j += 4) {
                    float x[2][4], y[2][4];
                    gen_load4<VEC>(x[0], D + j, dK - j);
                    gen_load4<VEC>(x[1], D + an + j, dK - j);
                    gen_load4<VEC>(y[0], dE + j, dK - j);   // dE is not written by this kernel
                    gen_load4<VEC>(y[1], dE + pn + j, dK - j);
#pragma unroll
                    for (int t = 0; t < 4; ++t)
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            acc[s][0] = fmaf(y[s][t], x[0][t], acc[s][0]);
                            acc[s][1] = fmaf(y[s][t], x[1][t], acc[s][1]);
                        }
                }
            }
#pragma unroll
            for (int s = 0; s < 2; ++s) { sum[s][0] += acc[s][0]; sum[s][1] += acc[s][1]; }
        }
        const float4 x = make_float4(sum[0][0], sum[0][1], sum[1][0], sum[1][1]);
        if (parts > 1) s_part[it] = x;               // then a thread has one item
        else add(ie, x);
    }
    if (parts > 1) {
        __syncthreads();
        if ((int)threadIdx.x < items) {
            float4 x = s_part[threadIdx.x];
            for (int part = 1; part < parts; ++part) {
                const float4 y = s_part[part * items + threadIdx.x];
                x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
            }
            add((int)threadIdx.x, x);
        }
    }
}
