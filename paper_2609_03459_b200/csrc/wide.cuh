// Sweeps of the shape with P_{K-2} of 8 rows and a slice of core K-1 of up to 64 x 256 (four cores, rank 64: C of 32 x 64).
//
// The intermediate product of one group is large (8 x 64 by 64 x 256) and its slice (64 KB) is shared by all groups of a
// run of the digit-major order, so a CTA of eight warps keeps the slice in shared memory and multiplies four groups (32
// stacked rows) at a time: a warp owns 32 columns, and every fragment of the slice that it loads and splits serves two row
// tiles.  Rows are then dealt out to the warps.  Two CTAs fit an SM (109 KB each): one multiplies while the other streams
// last-core slices.  22 k groups, 61 k rows: forward sweep 417 us with a pair of groups per CTA and the look-ups in line, 205 us
// now (3xTF32 products alone: 65 us at the mma.sync rate; the rest is the barriers around them and the rows' round trips);
// backward sweep of 4.7 k groups 135 -> 90 us.
#pragma once
#include "common.cuh"
#include "mma.cuh"

#define WIDE_THREADS 256
#define WIDE_GROUPS 4
#define WIDE_BP 264    // pitches in floats: fragment loads touch 32 different banks
#define WIDE_AP 68
#define WIDE_CP 68     // C as [32 rows p][64 values b]
#define WIDE_SMEM ((64 * WIDE_BP + 8 * WIDE_GROUPS * WIDE_AP + WIDE_GROUPS * 32 * WIDE_CP) * sizeof(float))

struct WideBatch {
    uint32_t g[WIDE_GROUPS], val[WIDE_GROUPS], im[WIDE_GROUPS], u0[WIDE_GROUPS], u1[WIDE_GROUPS];
    const float* left[WIDE_GROUPS];
};

// The batches of a work unit: next() leaves C of the current batch in Cs.  A batch's look-ups (digit-major list -> node ->
// prefix, rows, operand: a chain of dependent loads) run two batches ahead in the first four threads, its P and, at a run
// boundary, its slice are fetched while the rows of the batch before are made (P in registers: the space of As then holds
// the rows' operands).  Every thread calls next() the same number of times; As and Cs are free after it until the next call.
// ROUNDED: C's sums are rounded in fp32 after every k step (the backward, whose C was made with FMAs before; error of dG_K
// against 64 bits 5.6e-7 -> 3.4e-7, training call of 86 k lookups 743 -> 753 us).  The forward keeps the plain chain that it has always had.
template <bool ROUNDED>
struct WideLoop {
    const WsView& w;
    const TableDesc& td;
    WideBatch* const batches;      // [2], shared
    float *const Bs, *const As, *const Cs;
    uint32_t base, g1, held, node; // held: the slice in Bs; node (threads 0..3): this thread's group of batch + 1
    int cur;
    float4 p[2];                   // this thread's share of the next batch's P

    __device__ __forceinline__ WideLoop(const WsView& w_, const TableDesc& td_, uint2 rng, WideBatch* b, float* Bs_, float* As_, float* Cs_)
        : w(w_), td(td_), batches(b), Bs(Bs_), As(As_), Cs(Cs_), base(rng.x), g1(rng.y), held(0xffffffffu), cur(1)
    {
        if (base >= g1) return;
        node = list(base);
        WideBatch m;
        lookup(m);
        publish(m, 0);
        node = list(base + WIDE_GROUPS);
        __syncthreads();
        fetch(0);
    }
    __device__ __forceinline__ const WideBatch& batch() const { return batches[cur]; }
    // group at this thread's position of the batch at `pos` (none: 0xffffffff)
    __device__ __forceinline__ uint32_t list(uint32_t pos) const
    {
        if (threadIdx.x >= WIDE_GROUPS || pos + threadIdx.x >= g1) return 0xffffffffu;
        return tt_digit_major(w) ? w.tnode[w.K - 1][pos + threadIdx.x] : pos + threadIdx.x;
    }
    __device__ __forceinline__ void lookup(WideBatch& m) const   // of `node`, into this thread's registers (entry 0)
    {
        const int K = w.K;
        m.im[0] = 0xffffffffu;
        m.u0[0] = m.u1[0] = 0;
        m.g[0] = m.val[0] = 0;
        m.left[0] = nullptr;
        if (threadIdx.x >= WIDE_GROUPS || node == 0xffffffffu) return;
        m.g[0] = node;
        m.val[0] = w.val[K - 1][node];
        m.u0[0] = w.cstart[K - 1][node];
        m.u1[0] = w.cstart[K - 1][node + 1];
        m.left[0] = tt_left_operand(w, td, K - 1, node);
        m.im[0] = m.val[0] % (uint32_t)td.n[K - 2];
    }
    __device__ __forceinline__ void publish(const WideBatch& m, int slot)
    {
        if (threadIdx.x >= WIDE_GROUPS) return;
        WideBatch& b = batches[slot];
        const int q = threadIdx.x;
        b.g[q] = m.g[0]; b.val[q] = m.val[0]; b.im[q] = m.im[0]; b.u0[q] = m.u0[0]; b.u1[q] = m.u1[0]; b.left[q] = m.left[0];
    }
    __device__ __forceinline__ void slice(uint32_t im)
    {
        const int km = w.K - 2, ra = td.r[km];
        const float* B = td.core[km] + (size_t)im * td.slice_floats[km];
        for (int i = threadIdx.x; i < 64 * 64; i += WIDE_THREADS) {
            const int k = i >> 6, c = (i & 63) * 4;
            if (k < ra) tt_cp_async16(Bs + k * WIDE_BP + c, B + (size_t)k * 256 + c);
            else *reinterpret_cast<float4*>(Bs + k * WIDE_BP + c) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        held = im;
    }
    // P of the batch in `slot` into registers (columns past r_{K-2} zero), its first slice into Bs
    __device__ __forceinline__ void fetch(int slot)
    {
        const WideBatch& b = batches[slot];
        const int ra = td.r[w.K - 2];
        if (b.im[0] != 0xffffffffu && b.im[0] != held) slice(b.im[0]);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int i = threadIdx.x + x * WIDE_THREADS, row = i >> 4, c = (i & 15) * 4, q = row >> 3;
            p[x] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (b.im[q] == 0xffffffffu || c >= ra) continue;
            const float* src = b.left[q] + (row & 7) * ra + c;
            if ((ra & 3) == 0) p[x] = __ldg(reinterpret_cast<const float4*>(src));
            else {
                p[x].x = __ldg(src);
                if (c + 1 < ra) p[x].y = __ldg(src + 1);
                if (c + 2 < ra) p[x].z = __ldg(src + 2);
                if (c + 3 < ra) p[x].w = __ldg(src + 3);
            }
        }
    }
    __device__ __forceinline__ bool next()
    {
        if (base >= g1) return false;
        __syncthreads();             // the rows of the batch before are done with As and Cs
        cur ^= 1;
        const WideBatch& b = batches[cur];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int i = threadIdx.x + x * WIDE_THREADS;
            *reinterpret_cast<float4*>(As + (i >> 4) * WIDE_AP + (i & 15) * 4) = p[x];
        }
        WideBatch m;
        lookup(m);                   // batch + 1, in flight during the product
        node = list(base + 2 * WIDE_GROUPS);
        unsigned todo = 0;
#pragma unroll
        for (int q = 0; q < WIDE_GROUPS; ++q) todo |= b.im[q] != 0xffffffffu ? 1u << q : 0u;
        while (todo) {               // one pass per slice among the groups (more than one at a run boundary only)
            const uint32_t im = b.im[__ffs(todo) - 1];
            unsigned sel = 0;
#pragma unroll
            for (int q = 0; q < WIDE_GROUPS; ++q) sel |= b.im[q] == im ? 1u << q : 0u;
            todo &= ~sel;
            if (im != held) slice(im);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            product(sel);
            if (!todo) publish(m, cur ^ 1);
            __syncthreads();
        }
        base += WIDE_GROUPS;
        if (base < g1) fetch(cur ^ 1);
        return true;
    }
    __device__ __forceinline__ void product(unsigned sel)
    {
        const int ra = td.r[w.K - 2], lane = threadIdx.x & 31, wid = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
        float acc[2][4][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[mt][nt][x] = 0.f;
        const float* A = As + g * WIDE_AP + t;
        const float* B = Bs + t * WIDE_BP + 32 * wid + g;
#pragma unroll 2
        for (int k = 0; k < 64; k += 8) {
            if (k >= ra) break;
            Tf32Pair a[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                a[mt][0] = tt_split_tf32(A[16 * mt * WIDE_AP + k]);
                a[mt][1] = tt_split_tf32(A[(16 * mt + 8) * WIDE_AP + k]);
                a[mt][2] = tt_split_tf32(A[16 * mt * WIDE_AP + k + 4]);
                a[mt][3] = tt_split_tf32(A[(16 * mt + 8) * WIDE_AP + k + 4]);
            }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                Tf32Pair f[2];
                f[0] = tt_split_tf32(B[k * WIDE_BP + 8 * nt]);
                f[1] = tt_split_tf32(B[(k + 4) * WIDE_BP + 8 * nt]);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
                    if (ROUNDED) tt_mma_3xtf32_rounded(acc[mt][nt], a[mt], f);
                    else tt_mma_3xtf32(acc[mt][nt], a[mt], f);
            }
        }
        // stacked row 16 mt + 8 h + g: row g of P of group 2 mt + h; column c of the slice: row c / 64 under it, value c % 64
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!((sel >> (2 * mt + h)) & 1u)) continue;
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    const int c = 32 * wid + 8 * nt + 2 * t;
                    *reinterpret_cast<float2*>(Cs + (2 * mt + h) * (32 * WIDE_CP) + (4 * g + (c >> 6)) * WIDE_CP + (c & 63)) =
                        make_float2(acc[mt][nt][2 * h], acc[mt][nt][2 * h + 1]);
                }
            }
    }
};

// the group of row r of the batch, and its slot
__device__ __forceinline__ int wide_row(const WideBatch& b, uint32_t r, uint32_t& u)
{
    int q = 0;
    while (q < WIDE_GROUPS - 1 && r >= b.u1[q] - b.u0[q]) r -= b.u1[q] - b.u0[q++];
    u = b.u0[q] + r;
    return q;
}
__device__ __forceinline__ uint32_t wide_rows(const WideBatch& b)
{
    uint32_t n = 0;
#pragma unroll
    for (int q = 0; q < WIDE_GROUPS; ++q) n += b.u1[q] - b.u0[q];
    return n;
}
