// The rows of a batch of groups as one stream of steps (four rows of one group each) that a warp fetches ahead of its products.
//
// A warp that loads a pair of rows (last digits, then slices of the last core and rows of dE), multiplies them and goes on to the
// next pair waits for a chain of L2 round trips per pair; registers for a pair of look-ahead cost more warps than they save.  Here
// the rows come through a ring in shared memory (cp.async, no registers), across the groups of the batch, and the last digits eight
// steps ahead of that.  Backward sweeps, loop over pairs / stream, us: rank 16, C of 16 rows: 8 tables x 0.47 M rows 190 / 166, x
// 2.06 M rows 430 / 379; C of 16 rows, rank 8 (8 tables, 5 M lookups) 233 / 201; 8 rows, rank 16 328 / 217; 4 rows, rank 32 379 /
// 326; 4 rows, rank 16 287 / 205, weighted, 4 M lookups 242 / 177; the sweeps of the 60-table step together 7.05 / 6.88 ms.  Bound
// by instruction latency at 16 to 20 warps per SM (rank 16, 0.47 M rows: issue slots 40 %, LSU 43 %, L1 48 %, tensor pipe 20 %) and
// by the end of the grid.  A ring of three steps is no faster, more warps at the price of spills are slower (rank 16 at 96
// registers 404 against 377).  With C of 16 x 32 or 8 x 32 its 9 KB of C tiles per warp leave twelve warps per SM: 685 against 668
// and 567 against 522, so those shapes keep the loop without a ring, and so do all forward sweeps, whose row stage has half the
// operands (rank 32 373 against 328, rank 16 232 against 176). Where groups hold one to four rows each, the loop over pairs with
// its 24 warps is the faster one (8 tables of 40 M rows, 0.66 M spread lookups: rank 16, C of 16 rows 404 / 498; 4 rows, rank 32
// 386 / 496; 8 and 4 rows, rank 16 323 / 345, 249 / 283; training calls 1353 / 1444, 1353 / 1462, 1058 / 1070, 894 / 920).  As a
// kernel of its own for tables of few and even rows it gave those calls 2 to 5 % and took up to 10 % of calls over tables of mixed
// sizes, which the stream serves better than either (8 tables of 10 k to 40 M rows, 0.25 M spread lookups, call: pairs 347, stream
// 328, both 346).
#pragma once
#include "common.cuh"

// 16-byte asynchronous copy global -> shared (32-bit address), past L1; zeros instead of the source where !some
__device__ __forceinline__ void tt_cp_async16_or_zero(uint32_t smem_dst, const void* gsrc, bool some)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gsrc), "r"(some ? 16u : 0u) : "memory");
}

// PM x RB: C of a group; NG: groups of a batch; PD: steps in the ring
template <int PM, int RB, int NG, int PD>
struct RowStream {
    // pitches of a row of dE and of a slice: 8 (or 24) floats past a multiple of 32, so that four rows lie in different banks
    static constexpr int EP = PM * 4 + 8;
    static constexpr int DP = RB * 4 + 8;
    static constexpr int STEP = 4 * EP + 4 * DP;        // floats per ring slot
    static constexpr int INFO = 2 * 48 + 5 * 8;         // words: two blocks of eight steps, the groups
    static constexpr int FLOATS = PD * STEP + INFO;

    const uint32_t* __restrict__ rows;
    const float* __restrict__ GK;      // last core, with this lane's offset in a slice
    float* ring;
    uint32_t ring_s;                   // its shared address
    uint32_t steps, next;              // of the batch; the next one to stage
    uint32_t nid, nuf, nqn;            // lane: row slot of the block (eight steps) after the one that is being staged

    __device__ __forceinline__ RowStream(const uint32_t* rows_, const float* GK_, float* ring_, int lane)
        : rows(rows_), GK(GK_ + 4 * (lane % RB)), ring(ring_), ring_s((uint32_t)__cvta_generic_to_shared(ring_))
    {
    }
    // of step s: last digits of its rows, first row, group | rows << 8
    __device__ __forceinline__ uint32_t* ids(uint32_t s) const { return reinterpret_cast<uint32_t*>(ring + PD * STEP) + 48 * ((s >> 3) & 1) + 4 * (s & 7); }
    __device__ __forceinline__ uint32_t* first(uint32_t s) const { return reinterpret_cast<uint32_t*>(ring + PD * STEP) + 48 * ((s >> 3) & 1) + 32 + (s & 7); }
    __device__ __forceinline__ uint32_t* group_rows(uint32_t s) const { return first(s) + 8; }
    __device__ __forceinline__ uint32_t* groups() const { return reinterpret_cast<uint32_t*>(ring + PD * STEP) + 96; }   // [5][8]: end, u0, u1, row base, node

    __device__ __forceinline__ void look_up(uint32_t b, int lane)
    {
        const uint32_t s = 8 * b + (lane >> 2);
        if (8 * b >= steps) return;
        const uint32_t* gr = groups();
        uint32_t k = 0, start = 0;
#pragma unroll
        for (int i = 0; i < NG; ++i) {
            const uint32_t e = gr[i];
            if (e <= s) { k = i + 1; start = e; }
        }
        nqn = 0; nuf = 0; nid = 0;
        if (k < NG) {
            const uint32_t e1 = gr[16 + k];
            nuf = gr[8 + k] + 4 * (s - start);
            nqn = k | (min(4u, e1 - nuf) << 8);
            nid = __ldg(rows + min(nuf + (lane & 3), e1 - 1)) - gr[24 + k];   // (past the last row: the last one again)
        }
    }
    // the block that was looked up becomes the one to stage
    __device__ __forceinline__ void publish(uint32_t b, int lane)
    {
        ids(8 * b)[lane] = nid;
        if ((lane & 3) == 0) { first(8 * b)[lane >> 2] = nuf; group_rows(8 * b)[lane >> 2] = nqn; }
        __syncwarp();
        look_up(b + 1, lane);
    }
    // lane k < cnt: rows [u0, u1) of group k and the row id of its first possible row
    __device__ __forceinline__ void begin(uint32_t node, uint32_t u0, uint32_t u1, uint32_t row_base, int lane)
    {
        uint32_t end = (u1 - u0 + 3) >> 2;
#pragma unroll
        for (int o = 1; o < NG; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += y;
        }
        steps = __shfl_sync(0xffffffffu, end, NG - 1);
        next = 0;
        uint32_t* gr = groups();
        if (lane < NG) { gr[lane] = end; gr[8 + lane] = u0; gr[16 + lane] = u1; gr[24 + lane] = row_base; gr[32 + lane] = node; }
        __syncwarp();
        look_up(0, lane);
    }
    // starts the first PD steps
    __device__ __forceinline__ void fill(const float* __restrict__ E, int lane)
    {
#pragma unroll 1
        for (int i = 0; i < PD; ++i) stage(i, E, lane);
    }
    // the next step into ring slot `slot`; E: the rows of dE
    __device__ __forceinline__ void stage(int slot, const float* __restrict__ E, int lane)
    {
        if (next < steps) {
            if ((next & 7) == 0) publish(next >> 3, lane);
            const uint32_t dst = ring_s + slot * (STEP * 4);
            const uint32_t* id = ids(next) + lane / RB;
            const uint32_t uf = *first(next), nr = *group_rows(next) >> 8;
            const float* src = E + (size_t)uf * (PM * 4) + 4 * lane;
#pragma unroll
            for (int x = 0; x < (4 * PM + 31) / 32; ++x) {
                const int r = lane / PM + x * (32 / PM);
                const bool ok = (uint32_t)r < nr;
                if (PM >= 8 || lane < 16) tt_cp_async16_or_zero(dst + (r * EP + 4 * (lane % PM)) * 4, src + (ok ? 128 * x : -4 * lane), ok);
            }
#pragma unroll
            for (int x = 0; x < 4 * RB / 32; ++x) {
                const int r = lane / RB + x * (32 / RB);
                const uint32_t to = dst + (4 * EP + r * DP + 4 * (lane % RB)) * 4;
                const float* from = GK + (size_t)id[x * (32 / RB)] * (RB * 4);
                tt_cp_async16_or_zero(to, from, (uint32_t)r < nr);
            }
            ++next;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // the oldest step in flight is in its slot
    __device__ __forceinline__ const float* wait(int slot) const
    {
        asm volatile("cp.async.wait_group %0;" ::"n"(PD - 1) : "memory");
        __syncwarp();
        return ring + slot * STEP;
    }
};

// the row of a step that lane group i (of four) owns in the products over columns (row, j): with pitches of 8 floats past a multiple
// of 32, rows 0 and 2, and 1 and 3, fill the banks of a 64-bit load's half warp
__device__ __forceinline__ int tt_stream_row(int i) { return ((i & 1) << 1) | (i >> 1); }

__device__ __forceinline__ void tt_red_v4_if(bool some, float* p, float x, float y, float z, float wv)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t@q red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(wv), "r"((unsigned)some) : "memory");
}
