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

// A bag of more than two pieces, to be summed by whoever is free: see k_direct
struct DirectBag {
    uint32_t bag, lo, hi;      // its lookups [lo, hi); none where the record is not used
    uint32_t base;             // its first piece among those of all such bags
    uint32_t next, blocks;     // next piece to be handed out; blocks of DIRECT_JOIN pieces that are summed
    uint32_t unused[2];
};
#define DIRECT_JOIN 32
// a warp's flags: as the bits of the status word; there were lookups; the team's bag is a long one
#define DIRECT_BAD_ID (uint32_t)TT_EMB_STATUS_INDEX
#define DIRECT_BAD_OFFSET (uint32_t)TT_EMB_STATUS_OFFSETS
#define DIRECT_LOOKUPS 16u
#define DIRECT_LONG 32u
#define DIRECT_NONE 0xffffffffu    // no record
#define DIRECT_WHOLE 0xfffffffeu   // a long bag that found no room: summed by its team alone
#define DIRECT_STAY 1500           // ns that a CTA whose bags are all empty waits for long bags to be found
// counters, from CTR_DIRECT on: CTAs that have reported (bit 31: there are long bags), their status bits, 2..5 for tt_regroup, next bag
#define DIRECT_PIECES 7            // pieces of all long bags
#define DIRECT_RECORDS 8           // 64 bits: records begun, and those that can be read
#define DIRECT_HELPED 10           // CTAs that have reported a second time
#define DIRECT_GONE 11             // 1 + those that had reported before there was a long bag

// a, p, c, d: floats of shared memory per warp for the slice of the first core, P_2 of four cores, C, the slice of the last core (KIND 3: a
// and p are the two buffers of direct_chunk); 1 << team_log warps make a bag
struct DirectPlan {
    int a, p, c, d, team_log, kind;
    uint32_t longest, piece;   // lookups of a bag that is not cut, at most, and of a piece of the others
    uint32_t scan;             // bags that a team looks through for longer ones, at most 32; 0: there can be none
    uint32_t most_pieces, most_bags;
    int64_t* offsets;          // in the row buffer, which this call does not use: copies for tt_regroup,
    void* ids;
    DirectBag* bags;           // [most_bags],
    uint32_t* arrived;         // [most_pieces] pieces of a block that are stored,
    float* sums;               // [most_pieces][D]
};

__device__ __forceinline__ unsigned long long* direct_records(uint32_t* ctr) { return reinterpret_cast<unsigned long long*>(ctr + DIRECT_RECORDS); }

// A record for bag `bag` of [lo, hi), by one thread: where it is, or DIRECT_WHOLE
__device__ __noinline__ uint32_t direct_announce(uint32_t* ctr, const DirectPlan& plan, uint32_t bag, uint32_t lo, uint32_t hi)
{
    const uint32_t n = (hi - lo + plan.piece - 1) / plan.piece;
    const uint32_t gone = atomicOr(ctr, 1u << 31), i = (uint32_t)atomicAdd(direct_records(ctr), 1ull), base = atomicAdd(ctr + DIRECT_PIECES, n);
    if (gone >> 31 == 0u) ctr[DIRECT_GONE] = 1u + gone;
    const bool room = i < plan.most_bags && base < plan.most_pieces && n <= plan.most_pieces - base;   // (with well-formed offsets always)
    if (i < plan.most_bags) {
        DirectBag r = {bag, lo, room ? hi : lo, base, 0u, 0u, {0u, 0u}};
        plan.bags[i] = r;
    }
    if (room)
        for (uint32_t x = 0; x < n; x += DIRECT_JOIN) plan.arrived[base + x / DIRECT_JOIN] = 0u;
    __threadfence();
    atomicAdd(direct_records(ctr), 1ull << 32);
    return room ? i : DIRECT_WHOLE;
}

// the next piece of record r, if there is one
__device__ __forceinline__ bool direct_claim(const DirectPlan& plan, uint32_t r, uint32_t& bag, uint32_t& lo, uint32_t& hi, int lane)
{
    DirectBag* const b = plan.bags + r;
    uint32_t x = 0;
    if (lane == 0) x = atomicAdd(&b->next, 1u);
    x = __shfl_sync(0xffffffffu, x, 0);
    const uint4 of = __ldcg(reinterpret_cast<const uint4*>(b));
    if (x >= (of.z - of.y + plan.piece - 1) / plan.piece) return false;
    bag = of.x;
    lo = of.y + x * plan.piece;
    hi = min(lo + plan.piece, of.z);
    return true;
}

// A piece of a long bag for a warp: of the bags that its team has found (own[lane], bag bag0 + lane; null for all but its first warp),
// which nobody else may have seen, then of any.  DIRECT_NONE: there is none, otherwise its record; DIRECT_WHOLE: a bag as a whole.
__device__ __forceinline__ uint4 direct_find(const WsView& w, const DirectPlan& plan, uint32_t* own, uint32_t bag0, int lane)
{
    uint32_t bag = 0, lo = 0, hi = 0;
    while (own) {
        const uint32_t mine = own[lane];
        const unsigned have = __ballot_sync(0xffffffffu, mine != DIRECT_NONE);
        if (!have) break;
        const int src = __ffs(have) - 1;
        const uint32_t rec = __shfl_sync(0xffffffffu, mine, src);
        bool got = false;
        if (rec == DIRECT_WHOLE) {
            bag = bag0 + src;
            const int64_t o = __ldg(w.offsets + bag), o_next = __ldg(w.offsets + bag + 1);
            lo = o < 0 ? 0u : (uint32_t)o;
            hi = o_next > w.L ? (uint32_t)w.L : (uint32_t)o_next;
        } else got = direct_claim(plan, rec, bag, lo, hi, lane);
        if (!got && lane == src) own[lane] = DIRECT_NONE;
        __syncwarp();
        if (got || rec == DIRECT_WHOLE) return make_uint4(bag, lo, hi, rec);
    }
    for (int tries = 0; tries < 64; ++tries) {
        const unsigned long long records = __ldcg(direct_records(w.counters + CTR_DIRECT));
        uint32_t n = (uint32_t)records;
        if (n != 0 && (uint32_t)(records >> 32) == n) {    // all that are begun can be read
            __threadfence();
            n = min(n, plan.most_bags);
            const uint32_t first = (blockIdx.x * DIRECT_WARPS + (threadIdx.x >> 5)) % n;   // not all teams the same one
            for (uint32_t i = lane; i - lane < n; i += 32) {
                uint32_t r = first + i;
                if (r >= n) r -= n;
                for (;;) {
                    bool open = false;
                    if (i < n) {
                        const uint4 of = __ldcg(reinterpret_cast<const uint4*>(plan.bags + r));
                        open = (uint64_t)__ldcg(&plan.bags[r].next) * plan.piece < of.z - of.y;
                    }
                    const unsigned any = __ballot_sync(0xffffffffu, open);
                    if (!any) break;
                    const uint32_t rec = __shfl_sync(0xffffffffu, r, __ffs(any) - 1);
                    if (direct_claim(plan, rec, bag, lo, hi, lane)) return make_uint4(bag, lo, hi, rec);
                }
            }
            break;
        }
    }
    return make_uint4(0u, 0u, 0u, DIRECT_NONE);
}

// sum = pieces 0, step, 2 step, .. (n of them) at src in order; a lane's columns as in k_direct
__device__ __forceinline__ void direct_sum(float (&sum)[4], const float* src, uint32_t n, uint32_t step, int D, bool quads, int lane)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) sum[i] = 0.f;
    if (quads) {
        if (4 * lane >= D) return;
#pragma unroll 8
        for (uint32_t x = 0; x < n; ++x) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(src + (size_t)x * step * D) + lane);
            sum[0] += v.x; sum[1] += v.y; sum[2] += v.z; sum[3] += v.w;
        }
    } else
        for (uint32_t x = 0; x < n; ++x)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (lane + 32 * i < D) sum[i] += __ldcg(src + (size_t)x * step * D + lane + 32 * i);
}
__device__ __forceinline__ void direct_store(float* dst, const float (&sum)[4], int D, bool quads, int lane)
{
    if (quads) {
        if (4 * lane < D) *reinterpret_cast<float4*>(dst + 4 * lane) = make_float4(sum[0], sum[1], sum[2], sum[3]);
    } else
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (lane + 32 * i < D) dst[lane + 32 * i] = sum[i];
}
// The sum of a piece (of record item.w, from lookup item.y on) is done: true for the piece that arrives last, with the sum of all of them,
// in order (DIRECT_JOIN at a time by the last of those, then these sums), and the bag's length
__device__ __forceinline__ bool direct_join(const DirectPlan& plan, uint4 item, float (&sum)[4], int D, bool quads, uint32_t& len, int lane)
{
    DirectBag* const b = plan.bags + item.w;
    const uint4 of = __ldcg(reinterpret_cast<const uint4*>(b));
    len = of.z - of.y;
    const uint32_t n = (len + plan.piece - 1) / plan.piece, x = (item.y - of.y) / plan.piece, block = x / DIRECT_JOIN, blocks = (n + DIRECT_JOIN - 1) / DIRECT_JOIN;
    float* const at = plan.sums + (size_t)of.w * D;
    direct_store(at + (size_t)x * D, sum, D, quads, lane);
    __threadfence();
    __syncwarp();
    uint32_t seen = 0;
    if (lane == 0) seen = atomicAdd(plan.arrived + of.w + block, 1u);
    const uint32_t m = min((uint32_t)DIRECT_JOIN, n - block * DIRECT_JOIN);
    if (__shfl_sync(0xffffffffu, seen, 0) != m - 1) return false;
    __threadfence();
    direct_sum(sum, at + (size_t)block * DIRECT_JOIN * D, m, 1, D, quads, lane);
    if (blocks == 1) return true;
    direct_store(at + (size_t)block * DIRECT_JOIN * D, sum, D, quads, lane);
    __threadfence();
    __syncwarp();
    if (lane == 0) seen = atomicAdd(&b->blocks, 1u);
    if (__shfl_sync(0xffffffffu, seen, 0) != blocks - 1) return false;
    __threadfence();
    direct_sum(sum, at, blocks, DIRECT_JOIN, D, quads, lane);
    return true;
}

extern __shared__ __align__(16) float direct_smem[];   // the records of a team's long bags, then a buffer for every warp
__device__ __forceinline__ uint32_t* direct_own(uint32_t team) { return reinterpret_cast<uint32_t*>(direct_smem) + 32 * team; }
__device__ __forceinline__ float* direct_buffer(const DirectPlan& plan)
{
    return direct_smem + 32 * DIRECT_WARPS + (threadIdx.x >> 5) * (plan.a + plan.p + plan.c + plan.d);
}

// Sum of the rows of lookups lo + part, lo + part + W, .. of [lo, hi), of table td, by one warp; a lane's columns: four neighbouring ones
// (quads), otherwise every 32nd.  KEEP: between chunks the sum is in shared memory (keep, four floats of a lane): with it in registers
// direct_chunk spilled (2x4x4, rank 16, 85 k lookups 57 / 55 us).
template <int KIND, bool WT, bool KEEP>
__device__ __forceinline__ void direct_rows(const WsView& w, const DirectPlan& plan, const TableDesc& td, float* const As, uint32_t lo, uint32_t hi,
                                            uint32_t part_of, uint32_t W, float* keep, float (&sum)[4], bool& quads_out, uint32_t& flags)
{
    const int lane = threadIdx.x & 31, K = KIND == 3 ? 3 : w.K, D = w.D;
    float *const Ps = As + plan.a, *const Cs = Ps + plan.p, *const Ds = Cs + plan.c;
    if constexpr (KEEP) *reinterpret_cast<float4*>(keep) = make_float4(0.f, 0.f, 0.f, 0.f);
    else
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[i] = 0.f;
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
    const int q4 = dK >> 2, span = rK / splits;
    const bool on = lane < splits * items;
    const float* e_c = C;
    const float4* e_d = reinterpret_cast<const float4*>(Ds);
    if (quads && on) {
        const int item = lane % items, s = lane / items, p = item / q4;
        e_c += p * cp + s * span;
        e_d += s * span * q4 + item - p * q4;
    }
    quads_out = quads;
    for (uint32_t l0 = lo; l0 < hi; l0 += 32 * W) {
        const uint32_t l = l0 + part_of + W * lane;
        uint32_t q = 0;
        bool ok = false;
        float wt = 1.f;
        if (l < hi) {
            const int64_t id = tt_index<true>(w, l);
            if (w.idx32) reinterpret_cast<int32_t*>(plan.ids)[l] = (int32_t)id; else reinterpret_cast<int64_t*>(plan.ids)[l] = id;
            ok = id >= 0 && id < td.N;
            flags |= ok ? 0u : DIRECT_BAD_ID;
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
                    for (int x = 0; x < span; x += 4) {
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
        if constexpr (KEEP) {       // (between chunks in shared memory: the registers are short)
            float4* const at = reinterpret_cast<float4*>(keep);
            float4 v = *at;
            v.x += part[0]; v.y += part[1]; v.z += part[2]; v.w += part[3];
            *at = v;
        } else
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[i] += part[i];
    }
    if constexpr (KEEP) {
        const float4 v = *reinterpret_cast<const float4*>(keep);
        sum[0] = v.x; sum[1] = v.y; sum[2] = v.z; sum[3] = v.w;
    }
    // the pieces of the sums over r_{K-1} meet once per bag
    if (quads)
        for (int o = items; o < splits * items; o <<= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
}

template <bool WT>
__device__ __forceinline__ void direct_write(const WsView& w, float* __restrict__ out, uint32_t t, uint32_t b, float (&sum)[4], uint32_t len, bool quads, int lane)
{
    const int D = w.D, items = quads ? D / 4 : D;
    if (WT && w.pool_mean && len > 0) {
        const float inv = 1.f / (float)len;
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

// The team's share of the offsets, from bag0 on, by its first warp: a record for each long bag, into direct_own
__device__ __forceinline__ void direct_look(const WsView& w, const DirectPlan& plan, uint32_t team, uint32_t bag0)
{
    const int lane = threadIdx.x & 31;
    const uint32_t bag = bag0 + lane, nb = (uint32_t)(w.T * w.B);
    uint32_t rec = DIRECT_NONE;
    if (lane < plan.scan && bag < nb) {
        const int64_t o = __ldg(w.offsets + bag), o_next = __ldg(w.offsets + bag + 1);
        const uint32_t lo = o < 0 ? 0u : o > w.L ? (uint32_t)w.L : (uint32_t)o, hi = o_next < 0 ? 0u : o_next > w.L ? (uint32_t)w.L : (uint32_t)o_next;
        if (hi > lo && hi - lo > plan.longest) rec = direct_announce(w.counters + CTR_DIRECT, plan, bag, lo, hi);
    }
    direct_own(team)[lane] = rec;
    __syncwarp();
}

// Pieces of long bags, until all are taken, each by one warp; the flags of their lookups.  After direct_look, for the first warp of a team.
template <int KIND, bool WT>
__device__ __noinline__ uint32_t direct_pieces(const WsView& w, const DirectPlan& plan, float* __restrict__ out)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, D = w.D;
    const uint32_t per = DIRECT_WARPS >> plan.team_log, team = wid >> plan.team_log, bag0 = (blockIdx.x * per + team) * plan.scan;
    uint32_t* const own = (wid & ((1 << plan.team_log) - 1)) == 0 ? direct_own(team) : nullptr;
    uint32_t flags = 0;
    for (;;) {
        const uint4 item = direct_find(w, plan, own, bag0, lane);
        if (item.w == DIRECT_NONE) return flags;
        float sum[4];
        bool quads;
        const uint32_t t = item.x / (uint32_t)w.B;
        direct_rows<KIND, WT, false>(w, plan, w.tdesc[t], direct_buffer(plan), item.y, item.z, 0, 1, nullptr, sum, quads, flags);
        uint32_t len = item.z - item.y;
        if (item.w == DIRECT_WHOLE || direct_join(plan, item, sum, D, quads, len, lane)) direct_write<WT>(w, out, t, item.x - t * (uint32_t)w.B, sum, len, quads, lane);
    }
}

// KIND: 0 any shape; 1, 2: ranks and d_K multiples of four, 2: P_{K-2} of at most two rows; 3: direct_chunk's shapes.
// A bag's warps take its lookups in turn; their sums meet in shared memory, in order.  The bags after the first of every team of warps are
// handed out through a counter.  Offsets and row ids are checked on the way.
// How long a bag is only the offsets say, so bags of more than plan.longest lookups are left out at first.  Every team looks through its
// share of the offsets for them when it begins (a team with one bag when it meets it) and writes records of those that it finds.  A CTA
// whose bags are done reports, and sees with the report whether there are any; then its warps take pieces of them.  The last piece to
// arrive at a bag's end adds them up.  Nobody waits for another CTA: the team that found a bag makes all pieces that no other has taken.
// Calls with one long bag, us, left whole / cut (grouped): two tables, 60 k lookups, 57 k of them in one bag, rank 8 6300 / 75, rank 16
// 11 700 / 105 (2200); 40 k, 20 k in one, rank 16 8300 / 72 (910); 14 k, 2 k in one, rank 32 6000 / 100 (165); 30 k, 20 k in one, 2x4x4, rank 32 44 000 / 94
// (780); bag lengths of a power law (exponent 1.1, up to 5000), 46 k lookups, rank 8 1110 / 66 (280); 1 k lookups, all in one of 1 k bags 460 / 29 (186).
template <int KIND, bool WT>
__global__ void __launch_bounds__(DIRECT_THREADS, DIRECT_CTAS) k_direct(const __grid_constant__ WsView w, float* __restrict__ out, const __grid_constant__ DirectPlan plan)
{
    tt_pdl_enter();
    __shared__ __align__(16) float s_sum[2][DIRECT_WARPS][DIRECT_MOST_D];   // two bags in turn: one barrier per bag
    __shared__ uint32_t s_next[2][DIRECT_WARPS];
    __shared__ uint32_t s_flags[DIRECT_WARPS];
    __shared__ int s_then;                   // 0: done, 1: the last CTA is, 2: there are long bags
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t W = 1u << plan.team_log, part_of = wid & (W - 1), B = (uint32_t)w.B, nb = (uint32_t)(w.T * w.B), L = (uint32_t)w.L;
    const uint32_t per = DIRECT_WARPS >> plan.team_log;
    auto clampL = [&](int64_t x) { return x < 0 ? 0u : (x > w.L ? L : (uint32_t)x); };
    uint32_t* const ctr = w.counters + CTR_DIRECT;
    const uint32_t team = wid >> plan.team_log, teams = gridDim.x * per;
    uint32_t bag = blockIdx.x * per + team, flags = 0;
    if (plan.scan > 1 && part_of == 0) direct_look(w, plan, team, bag * plan.scan);
    for (int turn = 0; bag < nb; turn ^= 1) {
        // bags past the first of every team are handed out: their lengths differ
        uint32_t next = nb;
        if (nb > teams && part_of == 0 && lane == 0) next = teams + atomicAdd(ctr + 6, 1u);
        const int64_t o = __ldg(w.offsets + bag), o_next = __ldg(w.offsets + bag + 1);
        // (without branches, which would hold up the loads that follow until the offsets are there)
        const bool wrong = (o < 0) | (o > w.L) | (o_next < o) | ((bag == 0) & (o != 0)) | ((bag + 1 == nb) & (o_next != w.L));
        flags |= wrong ? DIRECT_BAD_OFFSET : 0u;
        if (part_of == 0 && lane < 2 && (lane == 0 || bag + 1 == nb)) plan.offsets[bag + lane] = lane == 0 ? o : o_next;
        const uint32_t lo = clampL(o), end = clampL(o_next), t = bag / B, b = bag - t * B;
        const bool long_bag = end > lo && end - lo > plan.longest;
        const uint32_t hi = long_bag ? lo : end;
        flags |= (end > lo ? DIRECT_LOOKUPS : 0u) | (long_bag ? DIRECT_LONG : 0u);
        float sum[4];
        bool quads;
        direct_rows<KIND, WT, true>(w, plan, w.tdesc[t], direct_buffer(plan), lo, hi, part_of, W, &s_sum[turn][wid][4 * lane], sum, quads, flags);
        if (W > 1) {    // the warps of the bag, in order
            float (*const sums)[DIRECT_MOST_D] = s_sum[turn] + wid;
            if (part_of > 0) {
                if (quads) {
                    if (4 * lane < w.D) *reinterpret_cast<float4*>(&sums[0][4 * lane]) = make_float4(sum[0], sum[1], sum[2], sum[3]);
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
        if (part_of == 0 && !long_bag) direct_write<WT>(w, out, t, b, sum, hi - lo, quads, lane);
        bag = next;
    }
    if (plan.scan == 1 && part_of == 0) {
        if (flags & DIRECT_LONG) direct_look(w, plan, team, blockIdx.x * per + team);
        else direct_own(team)[lane] = DIRECT_NONE;
    }
    for (bool pieces = false;; pieces = true) {
        // the CTA that reports last writes the status word
        const uint32_t warp_flags = __reduce_or_sync(0xffffffffu, flags);
        if (lane == 0) s_flags[wid] = warp_flags;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t all = 0;
#pragma unroll
            for (int i = 0; i < DIRECT_WARPS; ++i) all |= s_flags[i];
            const uint32_t bits = all & (DIRECT_BAD_ID | DIRECT_BAD_OFFSET);
            if (bits) atomicOr(ctr + 1, bits);
            if (plan.scan != 0 && !(all & DIRECT_LOOKUPS)) __nanosleep(DIRECT_STAY);
            __threadfence();
            if (!pieces) {
                const uint32_t before = atomicAdd(ctr, 1u);
                s_then = before >> 31 ? 2 : before == gridDim.x - 1;
            } else {
                const uint32_t before = atomicAdd(ctr + DIRECT_HELPED, 1u);
                __threadfence();
                const uint32_t gone = __ldcg(ctr + DIRECT_GONE);       // (written before its writer reports here)
                s_then = gone != 0 && before == gridDim.x - gone;
            }
        }
        __syncthreads();
        if (s_then != 2) break;
        flags = direct_pieces<KIND, WT>(w, plan, out) | DIRECT_LOOKUPS;
    }
    if (s_then != 1) return;
    // the last CTA leaves the counters of this kernel at zero
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
            if (w.idx32) reinterpret_cast<int32_t*>(plan.ids)[l] = (int32_t)id; else reinterpret_cast<int64_t*>(plan.ids)[l] = id;
            bad = bad || id < 0 || id >= w.tdesc[t].N;
        }
        all = TT_EMB_STATUS_OFFSETS | (__syncthreads_or(bad) ? TT_EMB_STATUS_INDEX : 0);
    }
    if (threadIdx.x == 0) {
        *w.status = (int32_t)all;
        ctr[0] = 0u;
        ctr[1] = 0u;
        ctr[2] = 1u;           // not grouped: tt_regroup
        ctr[3] = (uint32_t)w.B;
        ctr[4] = L;
        ctr[5] = (uint32_t)w.idx32;
        for (int i = 6; i <= DIRECT_GONE; ++i) ctr[i] = 0u;
    }
}

// The row buffer holds the copies of the offsets, then of the row ids, then what belongs to the long bags
static size_t direct_copy_bytes(const tt_emb* h) { return ((size_t)h->T * h->v.B + 1 + (size_t)h->v.L) * sizeof(int64_t); }

#define DIRECT_MOST_SMEM (100 << 10)
#define DIRECT_FEWEST_BAGS 64          // with fewer, one long bag keeps the call waiting
#define DIRECT_MOST_LOOKUPS (1 << 18)
#define DIRECT_PIECE_TIME 0.15          // shortest piece of a long bag, as a share of the grouped call's time
// Whether the call is made this way, and how: the time that it would take against that of the grouped path, both as fitted to forward
// calls of eleven shapes, 1 to 16 tables, 64 to 65536 bags each, 1 k to 0.2 M lookups (us).
//   here      a lookup takes the chip 0.3 ns and its products or slices, whichever is longer (4x4x4, rank 8 / 16 / 32: 0.47 / 0.83 / 2.6
//             ns; D = 128 4.8; four cores, rank 64 25), a bag 0.28 ns; and a warp makes its lookups one after the other (one table, 64 bags of 55
//             lookups, eight warps each, rank 16 / 32 / 64: 17 / 48 / 445 us), a bag of 1.6 times the average length among them.
//   grouped   36 to 84 us with 1 k lookups, by shape, and 0.28 ns for each of the others.
//   shared    shapes with a kernel of their own, with at most 2.5 rows in the tables for a lookup: the grouped call once more, and `here` with it, fitted to calls near the
//             line (1369 calls of 13 shapes, 1 to 40 tables of 300 to 40 M rows each, exponents 0.6 to 1.6).  Rank 8, us, here / grouped: eight tables
//             of 3 k rows, 0.16 M lookups, 4x4x4 72 / 58, 2x4x4 68 / 56; four of 3 k, 66 k bags of one 69 / 53; sixteen, 0.13 M lookups 82 / 60.  Of
//             these calls 76 took more than 1.02 of the grouped time (up to 1.4) without this term, 25 do with it (11 others would be faster here,
//             1.02 to 1.23): how often the rows repeat only the ids say.
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
    if (lookups > grouped || chain > grouped) return false;
    // The line above was drawn for rows spread over large tables.  With few rows for the lookups the grouped call is shorter.
    if (fast && rows <= 5 * w.L / 2) {
        const double row = products > bytes / 1.5 ? products : bytes / 1.5;
        const double shared = 52 + 0.08e-3 * (double)w.L + 0.05e-3 * (double)(w.L < rows ? w.L : rows) + 0.4 * h->T + (products < 45000 ? products / 1500 : 30);
        const double here = 5 + (double)w.L * (0.26e-3 + (row > 1700 ? row : 1700) / 8.5e6) + (double)nb * 0.4e-3;
        if (here > shared) return false;
    }
    // Long bags, and their pieces: a warp's share of an average bag and a quarter more at least, and long enough to be worth its claim and
    // its sum.  Twice as many in each of the bag's warps are left whole.  Pieces of 0.15 / 0.3 / 0.6 of the grouped time: rank 8, 57 k lookups in one bag 75 / 67 /
    // 84; 3x3x5, 10 k in one 70 / 94 / 146; rank 16, 20 k in one 72 / 72 / 86; power law, 46 k, rank 8 66 / 78 / 78.
    const uint64_t warps = 1u << plan.team_log;
    uint64_t piece = 1;
    while (piece * warps < 1.25 * bag || piece * (0.6 + products / 5000) < DIRECT_PIECE_TIME * grouped) piece *= 2;
    const size_t at = (direct_copy_bytes(h) + 15) & ~(size_t)15, room = (size_t)h->capU * h->D * sizeof(float);
    plan.longest = 0xffffffffu;
    for (; 2 * warps * piece < (uint64_t)w.L; piece *= 2) {
        // a bag of n > 2 pieces' lookups has at most 1.5 n of them, and at least 3
        plan.most_pieces = (uint32_t)(3 * (uint64_t)w.L / (2 * piece)) + 1;
        plan.most_bags = plan.most_pieces / 3 + 1;
        const size_t bags = plan.most_bags * sizeof(DirectBag), arrived = (plan.most_pieces * sizeof(uint32_t) + 15) & ~(size_t)15;
        if (at + bags + arrived + (size_t)plan.most_pieces * h->D * sizeof(float) > room) continue;
        plan.piece = (uint32_t)piece;
        plan.longest = (uint32_t)(2 * warps * piece);
        char* const base = reinterpret_cast<char*>(w.E) + at;
        plan.bags = reinterpret_cast<DirectBag*>(base);
        plan.arrived = reinterpret_cast<uint32_t*>(base + bags);
        plan.sums = reinterpret_cast<float*>(base + bags + arrived);
        break;
    }
    plan.offsets = reinterpret_cast<int64_t*>(w.E);
    plan.ids = plan.offsets + nb + 1;
    return true;
}

// launched: whether the call is made this way
cudaError_t tt_launch_direct(tt_emb* h, float* out, bool* launched, cudaStream_t s)
{
    const WsView& w = h->v;
    DirectPlan plan;
    *launched = false;
    if (!direct_plan(h, plan)) return cudaSuccess;
    const size_t smem = 32 * DIRECT_WARPS * sizeof(float) + (size_t)(plan.a + plan.p + plan.c + plan.d) * DIRECT_WARPS * sizeof(float);
    const bool wt = w.psw || w.pool_mean;
    auto kern = plan.kind == 3 ? (wt ? k_direct<3, true> : k_direct<3, false>) : plan.kind == 0 ? (wt ? k_direct<0, true> : k_direct<0, false>)
              : plan.kind == 1 ? (wt ? k_direct<1, true> : k_direct<1, false>) : (wt ? k_direct<2, true> : k_direct<2, false>);
    cudaError_t e;
    int& per_sm = h->direct_ctas[wt];     // kernel and shared memory are those of the handle's tables: asked once per bind
    if (per_sm == 0) {
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, DIRECT_MOST_SMEM + 32 * DIRECT_WARPS * (int)sizeof(float))) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, DIRECT_THREADS, smem)) != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
    }
    const int64_t nb = (int64_t)h->T * w.B, need = ((nb << plan.team_log) + DIRECT_WARPS - 1) / DIRECT_WARPS, most = (int64_t)h->sm_count * per_sm;
    const int64_t grid = need < most ? need : most, teams = grid * (DIRECT_WARPS >> plan.team_log);
    if (plan.longest != 0xffffffffu) plan.scan = (uint32_t)((nb + teams - 1) / teams);
    if (plan.scan > 32) return cudaSuccess;     // (a bag to a lane; so many bags are no faster here)
    *launched = true;
    if ((e = tt_launch_pdl(kern, dim3((unsigned)grid), dim3(DIRECT_THREADS), smem, s, w, out, plan)) != cudaSuccess) return e;
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
