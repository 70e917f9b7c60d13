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
#include "tiles.cuh"

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
template <int THREADS>
__device__ __forceinline__ void gen_batch_c(const WsView& w, const TableDesc& td, int cnt, const GenBatch& b, float* Cs)
{
    const int K = w.K, km = K - 2, Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb), tile = Pm * pitch;
    if (K >= 3) {
        constexpr int MB = 8;
        const int M = td.P[km], ra = td.r[km], dm = td.d[km], cols = dm * rb, mblocks = (M + MB - 1) / MB;
        for (int it = threadIdx.x; it < cnt * mblocks * cols; it += THREADS) {
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
        for (int it = threadIdx.x; it < cnt * Pm * rb; it += THREADS) {
            const int q = it / (Pm * rb), e = it - q * (Pm * rb), p = e / rb;
            Cs[q * tile + p * pitch + (e - p * rb)] = b.left[q][e];
        }
    }
    __syncthreads();
}

// look up rows r0 .. r0 + n of the batch, at most one per thread (ends with a barrier)
__device__ __forceinline__ void gen_rows(const WsView& w, const TableDesc& td, int cnt, uint32_t r0, int n, GenBatch& b)
{
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

// ---- backward with last dim factors of 1, 2, 3, 5, 6 or 7 (DK) ---------------------------------------------------------------------
//
// Rows of dE and slices of the last core are no whole float4s there, and the items above take one load for every product or two, each of a
// warp's lanes from another place.  Here a chunk's rows pass through shared memory (Es, odd pitch, read as whole lines), and a thread holds
// four values of r_{K-1} by all of d_K, whose slice parts are whole float4s where the slice is: 9 loads for 20 products in dG_K, 20 for 60
// in dC at d_K = 5.  Bound by shared-memory loads and the scattered loads of the slices.  Chunks hold few rows (8 groups of 1 to 8 rows),
// so CTAs are small: with 128 / 96 / 64 threads the sweep of 4 tables with 3x3x5, ranks 6 and 4, 1 M lookups, takes 97 / 106 / 125 us, 135
// with the items above; with units of enough rows (TT_UNIT_ROWS_ODD) 3 tables, 0.14 M lookups 76 -> 40, one table, 43 k 50 -> 31.
// Below GEN_ODD_LOOKUPS a unit's few rows leave most threads idle here too, and theirs is the longer chain: 0.9 k lookups, calls 109 above,
// 111 here, 15 k 132 / 133, 36 k 189 / 165.  In the forward sweep, whose rows would be staged on their way out, the items above stay:
// the first of these calls takes 439 us with them and 448 with staged rows, another with 0.19 M lookups 359 and 386.
#define GEN_ODD_LOOKUPS (1 << 14)
#define GEN_ODD_THREADS 128
#define GEN_STAGE_FLOATS 12288   // of the staged rows; fewer than GEN_STAGE_LEAST rows leave threads without one
#define GEN_STAGE_LEAST 64
#define GEN_P 3                  // rows of C that a thread takes at a time
__host__ __device__ __forceinline__ int gen_stage_pitch(int D) { return D | 1; }
__host__ __device__ __forceinline__ int gen_stage_rows(int D)
{
    const int n = GEN_STAGE_FLOATS / gen_stage_pitch(D);
    return n < GEN_ODD_THREADS ? n : GEN_ODD_THREADS;
}

// d = na x DK values of the slice part at p (VEC: four rows, 16-byte aligned)
template <int DK>
__device__ __forceinline__ void gen_part(float (&d)[4 * DK], const float* __restrict__ p, int na, bool vec)
{
    if (vec && na == 4) {
#pragma unroll
        for (int v = 0; v < DK; ++v) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p) + v);
            d[4 * v] = x.x; d[4 * v + 1] = x.y; d[4 * v + 2] = x.z; d[4 * v + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int f = 0; f < 4 * DK; ++f) d[f] = f < na * DK ? __ldg(p + f) : 0.f;
    }
}

// the n looked-up rows of dE into Es (ends with a barrier)
__device__ __forceinline__ void gen_stage(const WsView& w, int n, const GenBatch& b, float* Es)
{
    const int ep = gen_stage_pitch(w.D);
    for (int i = threadIdx.x >> 5; i < n; i += GEN_ODD_THREADS / 32)
        for (int e = threadIdx.x & 31; e < w.D; e += 32) tt_cp_async4(Es + i * ep + e, w.E + (size_t)b.u[i] * w.D + e);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
}

// dG_K[i_K] += C^T . dE of the staged rows, a thread four rows of a slice
template <int DK>
__device__ __forceinline__ void gen_slice_odd(const WsView& w, const TableDesc& td, int n, const GenBatch& b, const float* Cs, const float* Es, float* gk)
{
    const int K = w.K, Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb), slice = td.slice_floats[K - 1], ep = gen_stage_pitch(w.D);
    for (int it = threadIdx.x; it < n * ((rb + 3) / 4); it += GEN_ODD_THREADS) {
        const int i = it % n, a0 = it / n * 4, na = min(4, rb - a0);
        const float* c = Cs + b.q[i] * (Pm * pitch) + a0;
        const float* dE = Es + i * ep;
        float x[4 * DK];
#pragma unroll
        for (int f = 0; f < 4 * DK; ++f) x[f] = 0.f;
        for (int p = 0; p < Pm; ++p) {
            float e[DK];
#pragma unroll
            for (int j = 0; j < DK; ++j) e[j] = dE[p * DK + j];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float y = c[p * pitch + min(a, na - 1)];
#pragma unroll
                for (int j = 0; j < DK; ++j) x[a * DK + j] = fmaf(y, e[j], x[a * DK + j]);
            }
        }
        float* dst = gk + (size_t)b.iK[i] * slice + a0 * DK;
        if ((slice & 3) == 0 && na == 4) {
#pragma unroll
            for (int v = 0; v < DK; ++v) {
                const float y[4] = {x[4 * v], x[4 * v + 1], x[4 * v + 2], x[4 * v + 3]};
                gen_red4(dst + 4 * v, y);
            }
        } else {
#pragma unroll
            for (int f = 0; f < 4 * DK; ++f)
                if (f < na * DK) atomicAdd(dst + f, x[f]);
        }
    }
}

// dC += dE . G_K[i_K]^T over the staged rows, r0 the first of them: GEN_P by four elements of one group's dC to a thread, otherwise as
// gen_backward_dc; s_part [4 GEN_P][GEN_ODD_THREADS]
template <int DK>
__device__ __forceinline__ void gen_dc_odd(const WsView& w, const TableDesc& td, uint32_t r0, int n, const GenBatch& b, const float* Es, float* dCs, float* s_part)
{
    const int K = w.K, Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb), slice = td.slice_floats[K - 1], ep = gen_stage_pitch(w.D);
    const int q0 = (int)b.q[0], nq = (int)b.q[n - 1] - q0 + 1, ab = (rb + 3) / 4, per = (Pm + GEN_P - 1) / GEN_P * ab, items = nq * per;
    const int parts = items < GEN_ODD_THREADS ? min(16, GEN_ODD_THREADS / items) : 1;
    auto add = [&](int ie, const float (&x)[GEN_P][4]) {
        const int qq = ie / per, e = ie - qq * per, p = e / ab * GEN_P, a0 = (e - e / ab * ab) * 4;
        float* dst = dCs + (q0 + qq) * (Pm * pitch) + p * pitch + a0;
#pragma unroll
        for (int k = 0; k < GEN_P; ++k)
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (p + k < Pm && a0 + a < rb) dst[k * pitch + a] += x[k][a];
    };
    for (int it = threadIdx.x; it < items * parts; it += GEN_ODD_THREADS) {
        const int part = it / items, ie = it - part * items, qq = ie / per, e = ie - qq * per, p = e / ab * GEN_P, a0 = (e - e / ab * ab) * 4;
        const int q = q0 + qq, na = min(4, rb - a0);
        int i0 = b.row0[q] > r0 ? (int)(b.row0[q] - r0) : 0, i1 = min(n, (int)(b.row0[q + 1] - r0));
        const int len = (i1 - i0 + parts - 1) / parts;
        i0 += part * len;
        i1 = min(i1, i0 + len);
        int row[GEN_P];
        float sum[GEN_P][4];
#pragma unroll
        for (int k = 0; k < GEN_P; ++k) {
            row[k] = min(p + k, Pm - 1) * DK;
#pragma unroll
            for (int a = 0; a < 4; ++a) sum[k][a] = 0.f;
        }
        for (int ib = i0; ib < i1; ib += 8) {
            float acc[GEN_P][4];
#pragma unroll
            for (int k = 0; k < GEN_P; ++k)
#pragma unroll
                for (int a = 0; a < 4; ++a) acc[k][a] = 0.f;
            const int ie8 = min(i1, ib + 8);
            for (int i = ib; i < ie8; ++i) {
                float d[4 * DK];
                gen_part<DK>(d, td.core[K - 1] + (size_t)b.iK[i] * slice + a0 * DK, na, (slice & 3) == 0);
#pragma unroll
                for (int k = 0; k < GEN_P; ++k) {
                    const float* dE = Es + i * ep + row[k];
#pragma unroll
                    for (int j = 0; j < DK; ++j) {
                        const float y = dE[j];
#pragma unroll
                        for (int a = 0; a < 4; ++a) acc[k][a] = fmaf(y, d[a * DK + j], acc[k][a]);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < GEN_P; ++k)
#pragma unroll
                for (int a = 0; a < 4; ++a) sum[k][a] += acc[k][a];
        }
        if (parts > 1) {                             // then a thread has one item
#pragma unroll
            for (int k = 0; k < GEN_P; ++k)
#pragma unroll
                for (int a = 0; a < 4; ++a) s_part[(4 * k + a) * GEN_ODD_THREADS + it] = sum[k][a];
        } else add(ie, sum);
    }
    if (parts > 1) {
        __syncthreads();
        if ((int)threadIdx.x < items) {
            float x[GEN_P][4];
#pragma unroll
            for (int k = 0; k < GEN_P; ++k)
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const float* s = s_part + (4 * k + a) * GEN_ODD_THREADS + threadIdx.x;
                    x[k][a] = s[0];
                    for (int part = 1; part < parts; ++part) x[k][a] += s[part * items];
                }
            add((int)threadIdx.x, x);
        }
    }
}

// The last dim factor that all of the handle's any-shape tables have, where the call is for the code above (otherwise 0), and the floats of
// their C tiles of a batch
inline int gen_odd_factor(const tt_emb* h, int& c_floats)
{
    int dk = 0;
    c_floats = 0;
    for (int t = 0; t < h->T; ++t) {
        const TableDesc& td = h->tab[t];
        if (td.fast >= 0) continue;
        const int d = td.d[h->K - 1], tile = td.P[h->K - 1] * gen_pitch(td.r[h->K - 1]);
        const int n = GEN_C_FLOATS / tile < GEN_GROUPS ? GEN_C_FLOATS / tile : GEN_GROUPS;
        if (dk != 0 && d != dk) return 0;
        dk = d;
        if (n * tile > c_floats) c_floats = n * tile;
    }
    return dk < 8 && dk % 4 != 0 && h->v.L >= GEN_ODD_LOOKUPS && gen_stage_rows(h->D) >= GEN_STAGE_LEAST ? dk : 0;
}
