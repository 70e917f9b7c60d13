// Backward path (paper Sec. 3.2 backward, Eq. 2) and SGD.
//
//   1. sort:  the forward left one (slot, bag) pair per lookup; a counting sort by slot (counts, which give every pair its
//             rank in its row -> segment starts -> scatter of the bags) groups the lookups of every distinct row.  Hot rows
//             would serialise global atomics, so each CTA first aggregates the duplicates of its tile in shared memory (owner
//             tags) and issues one global atomic per aggregated row per tile.
//   2. dE:    segmented sum of grad_out rows over the sorted pairs.  Fixed-size chunks of sorted positions per
//             warp (skew-proof); segments that cross chunk borders leave partial sums, which the last warp to arrive,
//             or with many chunks a second kernel, adds in position order.
//   3. last level: per group, C is rebuilt in shared memory; every row contributes C^T.dE to the slice of
//             the last core it selects and dE.D^T to the group's dC (summed over the rows sharing C before
//             going up, Eq. 2; the sum is the k-loop of the tensor-core product, so dC is written once).
//             The last core's slices are accumulated with vector reductions into TT_STRIPES L2-resident
//             partial copies, which are then added in a fixed order (shared-memory fp32 atomics measured
//             at 2.6 per clock per SM on this part, too slow for a CTA-private copy).
//   4. middle cores: dP_{k-1} of a parent = sum over its (contiguous) children; the gradient of slice i_k
//             = sum over the level-k nodes with that digit, enumerated by a second, digit-major bitmap sort.
//             Each output has exactly one owner, which sums in sorted order: no atomics.  (K = 2 has no middle
//             cores; a first-core slice whose group is cut across work units gets its pieces by atomic additions.)
#include "common.cuh"
#include "scan.cuh"
#include "mma.cuh"
#include "quad_mid.cuh"
#include "group.cuh"
#include "generic.cuh"
#include "wide.cuh"
#include "tiles.cuh"
#include "rows.cuh"
#include "stream.cuh"
#include <type_traits>

#define HT_SIZE 4096
#define HT_TILE 2048
#define HT_EMPTY 0xffffffffu

// ---------------------------------------------------------------------------------------------- small utilities

// What the backward adds into or does not write whole: the counts of the sort, the partial copies of the last cores' gradients, the
// first cores' gradients (only the slices of present first digits are written later).  One kernel at the start: as a clear of the counts
// here, and a memset and a kernel between dE and the sweeps, the last two were 8 us of every call's chain (8 tables, 1.6 M lookups,
// training call 585 -> 577 us; 65 k lookups, four cores 414 -> 411).
__global__ void __launch_bounds__(256) k_bwd_clear(WsView w)
{
    tt_pdl_enter();
    const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    const int parts = gridDim.x >= (uint32_t)w.T ? (int)(gridDim.x / (uint32_t)w.T) : 1;   // CTAs per table
    int x = blockIdx.x;
    float* g0 = nullptr;
    int64_t floats = 0;
    if (x < parts * w.T) { g0 = w.tdesc[x % w.T].grad[0]; floats = w.tdesc[x % w.T].core_floats[0]; }   // (on their way during the clears below)
    const uint32_t n = w.counters[CTR_LEVEL0 + w.K] + 1u;
    for (uint32_t i = first; i < n; i += step) w.cnt[i] = 0u;
    for (uint32_t i = first; (uint64_t)i << w.de_chunk_log < (uint64_t)w.L; i += step) w.chunk_ctr[i] = 0u;
    float4* g4 = reinterpret_cast<float4*>(w.gpart);                 // every table's copy is a whole number of float4s
    const int64_t n4 = (int64_t)TT_STRIPES * w.gpart_stride / 4;
    for (int64_t i = first; i < n4; i += step) g4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    while (x < parts * w.T) {
        for (int64_t i = (int64_t)(x / w.T) * blockDim.x + threadIdx.x; i < floats; i += (int64_t)parts * blockDim.x) g0[i] = 0.f;
        x += gridDim.x;
        if (x < parts * w.T) { g0 = w.tdesc[x % w.T].grad[0]; floats = w.tdesc[x % w.T].core_floats[0]; }
    }
}

// Positions per warp (a power of two), and where the warps leave the pieces of segments that cross a chunk border.  A chunk is walked
// serially, so short batches want short chunks (1024 positions: 65 thousand lookups kept 64 warps busy) and long ones
// chunks that amortise the borders.  dE with 32 / 128 / 256 / 512 / 1024 positions per warp, us: 65 k lookups (D = 128,
// at least 160 there) 39 / 39 / 60 / 101 / 185; 0.5 M (D = 32) 33 / 31 / 42 / 62 / 103; 1.6 M (D = 64) 72 / 70 / 70 / 85 /
// 113; 4 M (D = 16) 173 / 122 / 121 / 142 / 173.
static void tt_de_partition(tt_emb* h)
{
    WsView& w = h->v;
    int64_t want = w.L / 2048 < 128 ? w.L / 2048 : 128;
    if (want < w.L / 32768) want = w.L / 32768;
    int log = 5;
    while ((2LL << log) <= want && (1 << log) < TT_DE_CHUNK) ++log;
    // the pieces of more than L / TT_DE_CHUNK chunks go where the unsorted pairs were (the sort has consumed them): 8 bytes
    // per lookup, so a chunk holds at least about D positions
    const uintptr_t u0 = (reinterpret_cast<uintptr_t>(w.upairs) + 15) & ~(uintptr_t)15;
    const size_t room = reinterpret_cast<uintptr_t>(w.upairs + h->max_lookups + 1) - u0;
    while ((1 << log) < TT_DE_CHUNK && (size_t)((w.L + (1LL << log) - 1) >> log) * 2 * h->D * sizeof(float) > room) ++log;
    w.carry = (1 << log) < TT_DE_CHUNK ? reinterpret_cast<float*>(u0) : h->carry;
    while (((w.L + (1LL << log) - 1) >> log) > TT_POOL_MAX_SHARES) ++log;   // the room for the chunks' first rows and counters
    w.de_chunk_log = (uint32_t)log;
    w.chunk_slot = reinterpret_cast<uint32_t*>(w.pool_bounds);   // (the pooling is done with its boundaries)
    w.chunk_ctr = w.chunk_slot + TT_POOL_MAX_SHARES + 1;
}

// ---------------------------------------------------------------------------------------------- 1. sort by slot

// A pair's place among the pairs of its row: cnt[slot] += occurrences, rank[l] = occurrences claimed before this one.  With the ranks
// from here the placing pass claims nothing.  (Two passes of claims, one to count and one to place: sort of 60 tables 2620 us, of 240
// 1590, of 4 M weighted pairs 173, of 0.5 M 47; now 1825, 1236, 109, 30.)
//
// Aggregation of a tile's duplicates without a probing hash table (two shared-memory atomics per pair made the
// shared-memory atomic unit the limit of the pass): every pair stores a tag (low key bits, its number in the tile)
// into bucket h(key) with a plain store; after a barrier the bucket holds the tag of one of its writers.  That pair
// owns the bucket.  A pair with the owner's key is a duplicate: it counts itself in extra[h] (the only shared-memory
// atomic left, and only duplicates issue it) and the owner makes one global atomic for all of them.  A pair with another
// key lost the bucket and goes to the global counter by itself.  h takes the key bits above bit 19 as they are, so that
// bucket and the 20 low bits together identify the key and a 32-bit tag is enough.
#define TT_SORT0_TILES 8
#define HT_LOW_BITS 20
#define HT_ID_BITS 11
__device__ __forceinline__ uint32_t* tt_sort_ranks(const WsView& w)
{
    return tt_weighted(w) ? reinterpret_cast<uint32_t*>(w.wsorted) : reinterpret_cast<uint32_t*>(w.pairs) + (w.upairs - w.pairs);
}
__global__ void __launch_bounds__(256) k_sort_count(WsView w)
{
    tt_pdl_enter();
    static_assert(HT_TILE == (1 << HT_ID_BITS) && HT_SIZE == (1 << (32 - HT_LOW_BITS)) && HT_LOW_BITS + HT_ID_BITS <= 32, "tag layout");
    const uint2* __restrict__ upairs = w.upairs;
    uint32_t* const rank = tt_sort_ranks(w);
    const uint32_t capK = w.cap[w.K];
    __shared__ uint32_t tag[HT_SIZE];
    __shared__ uint32_t extra[HT_SIZE];   // duplicates of the owner's key, then the owner's rank
    const int64_t L = w.L;
    const int64_t ntiles = (L + HT_TILE - 1) / HT_TILE;
    for (int i = threadIdx.x; i < HT_SIZE; i += blockDim.x) extra[i] = 0u;
    // the first barrier of the tile loop orders this before the first atomic on extra
    enum { ROLE_NONE = 0, ROLE_OWNER = 1, ROLE_DUP = 2 };
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        uint32_t key[HT_TILE / 256];
        uint32_t st[HT_TILE / 256];   // bucket (12 bits) | number among the duplicates (12 bits) << 12 | role << 24
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j) {
            const int64_t l = tile * HT_TILE + j * 256 + threadIdx.x;
            const uint2 pr = l < L ? __ldcs(upairs + l) : make_uint2(HT_EMPTY, 0u);
            key[j] = pr.x >= capK || (int64_t)pr.y >= w.B ? HT_EMPTY : pr.x;  // invalid lookup (or malformed offsets)
        }
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j) {
            if (key[j] == HT_EMPTY) continue;
            const uint32_t low = key[j] & ((1u << HT_LOW_BITS) - 1u);
            const uint32_t h = ((key[j] >> HT_LOW_BITS) ^ ((low * 2654435761u) >> HT_LOW_BITS)) & (HT_SIZE - 1);
            st[j] = h;
            tag[h] = (low << HT_ID_BITS) | (uint32_t)(j * 256 + threadIdx.x);
        }
        __syncthreads();
        uint32_t* const out = rank + tile * HT_TILE + threadIdx.x;
        uint32_t first[HT_TILE / 256];   // claims: all of a thread's are on their way before the first is looked at (60 tables 2160 -> 1870)
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j) {
            if (key[j] == HT_EMPTY) continue;
            const uint32_t low = key[j] & ((1u << HT_LOW_BITS) - 1u);
            const uint32_t h = st[j];
            const uint32_t tg = tag[h];
            if ((tg >> HT_ID_BITS) == low) {
                if ((tg & (HT_TILE - 1)) == (uint32_t)(j * 256 + threadIdx.x)) st[j] = h | (ROLE_OWNER << 24);
                else st[j] = h | ((atomicAdd(&extra[h], 1u) + 1u) << 12) | (ROLE_DUP << 24);
            } else first[j] = atomicAdd(&w.cnt[key[j]], 1u);   // another key holds the bucket
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j) {   // one global atomic per owner
            if (key[j] == HT_EMPTY || (st[j] >> 24) != ROLE_OWNER) continue;
            first[j] = atomicAdd(&w.cnt[key[j]], 1u + extra[st[j] & (HT_SIZE - 1)]);
        }
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j) {
            if (key[j] == HT_EMPTY || (st[j] >> 24) == ROLE_DUP) continue;
            if ((st[j] >> 24) == ROLE_OWNER) extra[st[j] & (HT_SIZE - 1)] = first[j];
            out[j * 256] = first[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j) {
            if (key[j] == HT_EMPTY || (st[j] >> 24) != ROLE_DUP) continue;
            out[j * 256] = extra[st[j] & (HT_SIZE - 1)] + ((st[j] >> 12) & 0xfffu);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < HT_TILE / 256; ++j)
            if (key[j] != HT_EMPTY && (st[j] >> 24) == ROLE_OWNER) extra[st[j] & (HT_SIZE - 1)] = 0u;
    }
}

// Counts -> segment starts in one kernel: a row's count becomes the sum of those before it in its tile, the CTA that reports last adds up
// the tiles (a ticket counter; nobody waits), and a start is the sum of both (tt_seg_start).  The row buffer still holds the rows: those
// without pairs (malformed offsets leave all their lookups out) are set to zero, as nothing else writes their dE.
#define CNT_TILE_LOG 12
struct CntTotal {
    const WsView& w;
    __device__ void total(uint32_t tot) const { w.cnt[w.counters[CTR_LEVEL0 + w.K]] = tot; }
};
__global__ void __launch_bounds__(256) k_seg_starts(WsView w)
{
    tt_pdl_enter();
    constexpr int TILE = 1 << CNT_TILE_LOG, ITEMS = TILE / 256;
    __shared__ uint32_t sm[34];
    __shared__ uint32_t sv[TILE + TILE / 32];
    __shared__ uint32_t ticket;
    const uint32_t n = w.counters[CTR_LEVEL0 + w.K], ntiles = (n + TILE - 1) >> CNT_TILE_LOG, base = blockIdx.x << CNT_TILE_LOG;
    if (n == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) w.cnt[0] = 0u;
        return;
    }
    if (blockIdx.x >= ntiles) return;
    const bool holes = *w.status & TT_EMB_STATUS_OFFSETS;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t i = base + (uint32_t)j * 256 + threadIdx.x;
        sv[tt_scan_pad(j * 256 + threadIdx.x)] = i < n ? w.cnt[i] : 0u;
    }
    __syncthreads();
    uint32_t mine[ITEMS], s = 0, tot;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) { mine[j] = sv[tt_scan_pad(threadIdx.x * ITEMS + j)]; s += mine[j]; }
    if (holes)
        for (uint32_t i = base + threadIdx.x; i < n && i < base + TILE; i += 256)
            if (sv[tt_scan_pad(i - base)] == 0u)
                for (int e = 0; e < w.D; ++e) w.E[(size_t)i * w.D + e] = 0.f;
    uint32_t ex = tt_block_excl_scan(s, sm, tot);
    if (threadIdx.x == 0) {
        w.scan_tmp[blockIdx.x] = tot;
        __threadfence();                                   // the sum is visible before the ticket is
        ticket = atomicAdd(w.counters + CTR_SCAN_TICKET, 1u);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) { sv[tt_scan_pad(threadIdx.x * ITEMS + j)] = ex; ex += mine[j]; }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t i = base + (uint32_t)j * 256 + threadIdx.x;
        if (i < n) w.cnt[i] = sv[tt_scan_pad(j * 256 + threadIdx.x)];
    }
    if (ticket != ntiles - 1) return;
    __threadfence();
    tt_scan_spine_cta(CntTotal{w}, w.scan_tmp, ntiles, sm);
    if (threadIdx.x == 0) w.counters[CTR_SCAN_TICKET] = 0u;
}
// first sorted position of row `slot` (the number of pairs for slot = U)
__device__ __forceinline__ uint32_t tt_seg_start(const WsView& w, uint32_t slot, uint32_t U)
{
    return w.cnt[slot] + (slot < U ? w.scan_tmp[slot >> CNT_TILE_LOG] : 0u);
}

// The bags in sorted order, with the pairs' factors where the pooling has any; the row of a position follows from the segment starts, so
// that only the rows of the chunks' first positions are written down (chunk_slot).  No atomics and no barriers: the places are known.
// Bound by the scattered stores.  With 2 / 4 / 8 pairs per thread: 60 tables sort 1898 / 1867 / 1875 us, 4 M weighted pairs 106 / 109 /
// 112, 0.5 M 30 / 30 / 34.
#define SORT_PLACE_PER 4
template <bool WT>
__global__ void __launch_bounds__(256) k_sort_place(WsView w)
{
    tt_pdl_enter();
    constexpr int PER = SORT_PLACE_PER;
    const uint32_t capK = w.cap[w.K], U = w.counters[CTR_LEVEL0 + w.K];
    const uint32_t* const rank = tt_sort_ranks(w);
    const int64_t l0 = (int64_t)blockIdx.x * (256 * PER) + threadIdx.x;
    uint2 pr[PER];
    uint32_t rk[PER];
    float a[PER];
    int t = 0;
    if (WT && w.pool_mean) t = tt_find_table64(w.tl_start, w.T, l0);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int64_t l = l0 + j * 256;
        pr[j] = l < w.L ? __ldcs(w.upairs + l) : make_uint2(HT_EMPTY, 0u);
        if (pr[j].x >= capK || (int64_t)pr[j].y >= w.B) pr[j].x = HT_EMPTY;
        rk[j] = pr[j].x != HT_EMPTY ? __ldcs(rank + l) : 0u;
        if (WT) {
            a[j] = w.psw && l < w.L ? __ldg(w.psw + l) : 1.f;
            if (w.pool_mean && pr[j].x != HT_EMPTY) {
                while (t + 1 < w.T && w.tl_start[t + 1] <= l) ++t;
                const int64_t gb = (int64_t)t * w.B + pr[j].y;
                const int64_t len = __ldg(w.offsets + gb + 1) - __ldg(w.offsets + gb);
                a[j] /= (float)(len > 0 ? len : 1);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < PER; ++j)
        if (pr[j].x != HT_EMPTY) rk[j] += tt_seg_start(w, pr[j].x, U);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (pr[j].x == HT_EMPTY) continue;
        if (WT) w.pairs[rk[j]] = make_uint2(pr[j].y, __float_as_uint(a[j]));
        else reinterpret_cast<uint32_t*>(w.pairs)[rk[j]] = pr[j].y;
        if ((rk[j] & ((1u << w.de_chunk_log) - 1u)) == 0u) w.chunk_slot[rk[j] >> w.de_chunk_log] = pr[j].x;
    }
}

cudaError_t tt_launch_bwd_sort(tt_emb* h, cudaStream_t s)
{
    WsView& w = h->v;
    const int zgrid = h->sm_count * 8;
    cudaError_t e;
    tt_de_partition(h);
    if ((e = tt_launch_pdl(k_bwd_clear, dim3(zgrid), dim3(256), 0, s, w)) != cudaSuccess) return e;
    tt_note_launch();
    const int64_t ntiles = (w.L + HT_TILE - 1) / HT_TILE;
    int per_sm = 0;   // a persistent grid sized to what is actually resident (no partial second wave)
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sort_count, 256, 0)) != cudaSuccess) return e;
    // the counting pass as a grid of more CTAs than fit at once, TT_SORT0_TILES tiles each: the block scheduler then
    // balances the tiles' very different costs (a tile of popular rows aggregates to a few claims, one of unpopular rows
    // makes two thousand).  Sort with 4 / 8 / 24 / 48 tiles per CTA, us: 60 tables 2003 / 1825 / 1867 / 1876, 240 tables 1357 / 1236 / 1289 /
    // 1440
    int64_t g = (int64_t)(per_sm < 1 ? 1 : per_sm) * h->sm_count;
    if (g > ntiles) g = ntiles;
    if (g < 1) g = 1;
    const int64_t many = (ntiles + TT_SORT0_TILES - 1) / TT_SORT0_TILES;
    if (many > g) g = many;
    if ((e = tt_launch_pdl(k_sort_count, dim3((unsigned)g), dim3(256), 0, s, w)) != cudaSuccess) return e;
    tt_note_launch();
    const int64_t rows = (int64_t)w.cap[w.K] < w.L ? (int64_t)w.cap[w.K] : w.L;
    if ((e = tt_launch_pdl(k_seg_starts, dim3((unsigned)((rows >> CNT_TILE_LOG) + 1)), dim3(256), 0, s, w)) != cudaSuccess) return e;
    tt_note_launch();
    if (w.L == 0) return cudaGetLastError();
    if ((e = tt_launch_pdl(tt_weighted(w) ? k_sort_place<true> : k_sort_place<false>, dim3((unsigned)((w.L + 256 * SORT_PLACE_PER - 1) / (256 * SORT_PLACE_PER))), dim3(256), 0, s, w)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- 2. dE

// lane l of the warp owns float4 chunks l, l+32, ... of a row (VEC) or floats l, l+32, ... (!VEC)
template <bool VEC, int CPL>
struct RowAcc {
    float v[VEC ? 4 * CPL : CPL];
    __device__ void clear()
    {
#pragma unroll
        for (int i = 0; i < (VEC ? 4 * CPL : CPL); ++i) v[i] = 0.f;
    }
    // v += a * row (a = 1 gives exactly v + row)
    __device__ void add_row(const float* __restrict__ row, int D, int lane, float a = 1.f)
    {
        if (VEC) {
            const float4* r4 = reinterpret_cast<const float4*>(row);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int ch = lane + c * 32;
                if (ch * 4 < D) {
                    const float4 x = __ldg(r4 + ch);
                    v[4 * c] = fmaf(a, x.x, v[4 * c]); v[4 * c + 1] = fmaf(a, x.y, v[4 * c + 1]);
                    v[4 * c + 2] = fmaf(a, x.z, v[4 * c + 2]); v[4 * c + 3] = fmaf(a, x.w, v[4 * c + 3]);
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int i = lane + c * 32;
                if (i < D) v[c] = fmaf(a, __ldg(row + i), v[c]);
            }
        }
    }
    // v += the first piece (CPL = 1) of a row in shared memory
    __device__ void add_shared(const void* x)
    {
        const float* f = reinterpret_cast<const float*>(x);
#pragma unroll
        for (int i = 0; i < (VEC ? 4 : 1); ++i) v[i] += f[i];
    }
    __device__ void store(float* __restrict__ row, int D, int lane) const
    {
        if (VEC) {
            float4* r4 = reinterpret_cast<float4*>(row);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int ch = lane + c * 32;
                if (ch * 4 < D) r4[ch] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int i = lane + c * 32;
                if (i < D) row[i] = v[c];
            }
        }
    }
};

#define DE_SPILL_LOG 1     // half a chunk
// The sorted positions of a warp's chunk, 32 at a time: rows from the segment starts, bags (and factors) as stored.  `rows` and
// then `fetch` are called once per batch; after them the loads of the batch that follows are on their way.
struct DePairs {
    const WsView& w;
    uint32_t U, total, a, b;       // rows, pairs; the chunk [a, b)
    uint32_t prev, next_slot;      // row of the position before the chunk if the chunk starts inside it; of the position after it
    uint32_t row0, from, till;     // row of the chunk's first position, its first position and the one after its last
    uint32_t s, v;                 // row of the last position looked at; start of row s + 1 + lane
    uint32_t bag;
    float factor;
    bool holes;                    // there may be rows without pairs

    __device__ __forceinline__ uint32_t start(uint32_t slot) const { return slot < U ? tt_seg_start(w, slot, U) : total; }
    __device__ __forceinline__ DePairs(const WsView& w_, int64_t chunk) : w(w_)
    {
        U = w.counters[CTR_LEVEL0 + w.K];
        total = w.cnt[U];
        holes = *w.status & TT_EMB_STATUS_OFFSETS;
        const int64_t a64 = chunk << w.de_chunk_log;
        a = a64 < total ? (uint32_t)a64 : total;
        b = min(a + (1u << w.de_chunk_log), total);
    }
    template <bool WT>
    __device__ __forceinline__ void fetch(uint32_t p, int lane)    // positions p + lane
    {
        v = start(s + 1 + lane);
        bag = 0u;
        factor = 1.f;
        if (p + lane < b) {
            if (WT) {
                const uint2 x = __ldcs(w.pairs + p + lane);
                bag = x.x;
                factor = __uint_as_float(x.y);
            } else bag = __ldcs(reinterpret_cast<const uint32_t*>(w.pairs) + p + lane);
        }
    }
    // Positions that a chunk takes of the next one to end its last segment, instead of leaving a piece of it there
    __device__ __forceinline__ uint32_t spill() const { return (1u << w.de_chunk_log) >> DE_SPILL_LOG; }
    // a < b before; afterwards a = b where the chunk before has taken all of this one's positions
    template <bool WT, bool JOIN>
    __device__ __forceinline__ void begin(int64_t chunk, int lane)
    {
        s = w.chunk_slot[chunk];
        next_slot = b < total ? w.chunk_slot[chunk + 1] : HT_EMPTY;
        fetch<WT>(a, lane);
        row0 = s;
        from = start(s);
        if (JOIN && b < total) {
            const uint32_t end = start(next_slot + 1u);
            if (start(next_slot) < b && end - b <= spill()) {
                b = end;
                next_slot = HT_EMPTY;
            }
        }
        till = __shfl_sync(0xffffffffu, v, 0);
        prev = HT_EMPTY;
        if (from < a) {
            if (JOIN && till - a <= spill()) {          // the chunk before ends it
                a = till;
                if (a >= b) return;
                int k;
                do {                            // (more than one: rows without pairs)
                    k = __popc(__ballot_sync(0xffffffffu, v <= a));
                    s += k;
                    v = start(s + 1 + lane);
                } while (k == 32);
                fetch<WT>(a, lane);
                row0 = s;
                from = a;
                till = __shfl_sync(0xffffffffu, v, 0);
            } else prev = s;
        }
    }
    // bit j: position p + j starts another row than the one before it (j < n); where rows without pairs may be among them (lookups that
    // malformed offsets leave out): false, `rows` then finds the rows, otherwise every start is one row further and s is the row of the last
    // position
    __device__ __forceinline__ bool starts(uint32_t p, int n, unsigned& bits)
    {
        bits = __reduce_or_sync(0xffffffffu, v - p < (uint32_t)n ? 1u << (v - p) : 0u);
        if (holes) return false;
        s += __popc(bits);
        return true;
    }
    // row of position p + lane (lane < n), all lanes: n positions from p on
    __device__ __forceinline__ uint32_t rows(uint32_t p, int n, int lane)
    {
        uint32_t row = s;
        for (;;) {
            int k = 0;             // starts among those of rows s + 1 .. s + 32 that are not past this position
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, v, k + step - 1) <= p + lane) k += step;
            if (__shfl_sync(0xffffffffu, v, k) <= p + lane) ++k;
            row += k;
            if (!__any_sync(0xffffffffu, k == 32 && lane < n)) break;
            s += 32;               // (32 rows of one pair each, or rows without pairs)
            v = start(s + 1 + lane);
        }
        s = __shfl_sync(0xffffffffu, row, n - 1);
        return lane < n ? row : HT_EMPTY;
    }
};

// Segments that cross chunk borders leave a piece per chunk: the head of a chunk (its first row, begun in an earlier one) or the tail (goes
// on in the next; a chunk inside one segment has a tail only).  With few chunks the warp whose piece arrives last adds them up, in order
// (counters; nobody waits); a popular row spans hundreds of chunks, so that pieces are added 32 at a time, by the last of the 32, and
// then those sums.  A short rest of a segment stays with the chunk before (DE_SPILL_LOG), which leaves the popular rows' pieces only.
// With many chunks the wait for the stores at the end of every warp costs more than the kernel that adds the pieces up afterwards
// (k_dE_fix).  dE, kernel afterwards / last arrival, us: 65 k lookups, D = 128 26 / 21; 0.5 M, D = 32 31 / 27; 1 M, D = 45 86 / 70; 1.6 M, D =
// 64 69 / 60; 3.7 M, D = 64 (29 k chunks): call 1548 / 1500; 2.4 M, D = 16 (19 k chunks) call 711 / 718; 4 M, D = 16 (32 k chunks) 118 / 121;
// 60 tables (97 k chunks) 2150 / 2235.  (Warps that take chunks from a counter, with the counts a chunk later: 60 tables 2640.)
#define DE_JOIN_CHUNKS 16384      // twice as many for rows of more than 32 floats
#define DE_JOIN 32
// fields of a chunk's counter: pieces of 32 that start in it, of the first ones of a segment that does, sums of 32 of that segment
#define DE_CTR_REST 0
#define DE_CTR_FIRST 6
#define DE_CTR_SUMS 12
// dst = the pieces of chunks x, x + step, .. (m of them) of the segment that ends in chunk c1
template <bool VEC>
__device__ __forceinline__ void de_sum(const WsView& w, float* dst, uint32_t x, uint32_t m, uint32_t step, uint32_t c1, int lane)
{
    using piece_t = typename std::conditional<VEC, float4, float>::type;
    constexpr int PF = VEC ? 4 : 1, NF = 8;
    const int D = w.D, cols = D / PF;
    int lpr = 32;
    while (lpr > 1 && lpr / 2 >= cols) lpr >>= 1;
    const uint32_t slots = 32u / lpr, slot = lane / lpr;
    for (int c0 = 0; c0 < cols; c0 += lpr) {
        const int c = c0 + lane % lpr;
        RowAcc<VEC, 1> sum;
        sum.clear();
        for (uint32_t i0 = slot; i0 < m; i0 += NF * slots) {
            piece_t v[NF];
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                const uint32_t i = i0 + k * slots, y = x + i * step;
                v[k] = i < m && c < cols ? __ldcg(reinterpret_cast<const piece_t*>(w.carry) + ((size_t)y * 2 + (y < c1 ? 1 : 0)) * cols + c) : piece_t{};
            }
            RowAcc<VEC, 1> part;
            part.clear();
#pragma unroll
            for (int k = 0; k < NF; ++k) part.add_shared(&v[k]);
#pragma unroll
            for (int k = 0; k < PF; ++k) sum.v[k] += part.v[k];
        }
        for (int o = lpr; o < 32; o <<= 1)
#pragma unroll
            for (int k = 0; k < PF; ++k) sum.v[k] += __shfl_xor_sync(0xffffffffu, sum.v[k], o);
        if (slot == 0 && c < cols) sum.store(dst + PF * c, PF, 0);
    }
}
template <bool VEC>
__device__ __forceinline__ void de_arrive(const WsView& w, uint32_t chunk, uint32_t row, uint32_t from, uint32_t till, uint32_t spill, int lane)
{
    uint32_t c1 = (till - 1u) >> w.de_chunk_log;
    if (till - (c1 << w.de_chunk_log) <= spill) --c1;     // (the segment goes on past a border: c1 > c0)
    const uint32_t c0 = from >> w.de_chunk_log, pieces = c1 - c0 + 1u;
    const uint32_t block = (chunk - c0) / DE_JOIN, x = c0 + block * DE_JOIN, m = min((uint32_t)DE_JOIN, pieces - block * DE_JOIN);
    const int shift = block == 0 ? DE_CTR_FIRST : DE_CTR_REST;
    uint32_t seen = 0;
    if (lane == 0) seen = atomicAdd(w.chunk_ctr + x, 1u << shift) >> shift & 63u;
    if (__shfl_sync(0xffffffffu, seen, 0) != m - 1u) return;
    __threadfence();
    float* const out = w.E + (size_t)row * w.D;
    const uint32_t sums = (pieces + DE_JOIN - 1u) / DE_JOIN;
    de_sum<VEC>(w, sums == 1 ? out : w.carry + ((size_t)x * 2 + (x < c1 ? 1 : 0)) * w.D, x, m, 1, c1, lane);
    if (sums == 1) return;
    __threadfence();
    __syncwarp();
    if (lane == 0) seen = atomicAdd(w.chunk_ctr + c0, 1u << DE_CTR_SUMS) >> DE_CTR_SUMS;
    if (__shfl_sync(0xffffffffu, seen, 0) != sums - 1u) return;
    __threadfence();
    de_sum<VEC>(w, out, c0, sums, DE_JOIN, c1, lane);
}
// a chunk's pieces are stored; cur: row of its last position
template <bool VEC>
__device__ __forceinline__ void de_finish(const WsView& w, const DePairs& pairs, int64_t chunk, uint32_t cur, int lane)
{
    const bool begun = pairs.prev == pairs.row0, goes_on = pairs.next_slot == cur && !(begun && cur == pairs.row0);
    if (!begun && !goes_on) return;
    __threadfence();
    __syncwarp();
    if (begun) de_arrive<VEC>(w, (uint32_t)chunk, pairs.row0, pairs.from, pairs.till, pairs.spill(), lane);
    if (goes_on) de_arrive<VEC>(w, (uint32_t)chunk, cur, (uint32_t)(chunk << w.de_chunk_log), pairs.start(cur + 1u), pairs.spill(), lane);
}

template <bool VEC, int CPL>
__global__ void __launch_bounds__(256) k_dE(WsView w, const float* __restrict__ grad_out)
{
    tt_pdl_enter();
    constexpr int NF = !VEC && CPL <= 4 ? 16 / CPL : 4;   // narrow rows: more of them in flight
    const int lane = threadIdx.x & 31;
    const int64_t chunk = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    DePairs pairs(w, chunk);
    if (pairs.a >= pairs.b) return;
    const int D = w.D;
    const size_t gstride = (size_t)w.T * D;
    const bool weighted = tt_weighted(w);
    if (weighted) pairs.begin<true, false>(chunk, lane); else pairs.begin<false, false>(chunk, lane);
    const uint32_t a = pairs.a, b = pairs.b;
    if (a >= b) return;
    const uint32_t prev = pairs.prev, next = pairs.next_slot;
    RowAcc<VEC, CPL> acc;
    acc.clear();
    uint32_t cur = pairs.s;
    int tcur = tt_find_table(w.tb[w.K], w.T, cur);
    bool seg_first = true;
    float* carry = w.carry + (size_t)chunk * 2 * D;
    for (uint32_t p0 = a; p0 < b; p0 += 32) {
        const uint2 mine = make_uint2(pairs.rows(p0, (int)min(32u, b - p0), lane), pairs.bag);
        const float wmine = pairs.factor;
        if (p0 + 32 < b) { if (weighted) pairs.fetch<true>(p0 + 32, lane); else pairs.fetch<false>(p0 + 32, lane); }
        const int n = (int)min(32u, b - p0);
        // NF rows of grad_out in flight at a time (their addresses need the table of each pair's slot; positions are
        // sorted, so the table changes rarely), then the rows are folded in position order
        const int tmine = lane < n ? tt_find_table_from(w.tb[w.K], w.T, mine.x, tcur) : tcur;
        for (int j0 = 0; j0 < n; j0 += NF) {
            RowAcc<VEC, CPL> rowv[NF];
#pragma unroll
            for (int jj = 0; jj < NF; ++jj) {
                const int j = min(j0 + jj, n - 1);
                const uint32_t bag = __shfl_sync(0xffffffffu, mine.y, j);
                const int tj = __shfl_sync(0xffffffffu, tmine, j);
                rowv[jj].clear();
                if (j0 + jj < n) rowv[jj].add_row(grad_out + (size_t)bag * gstride + (size_t)tj * D, D, lane, 1.f);
            }
#pragma unroll
            for (int jj = 0; jj < NF; ++jj) {
                const int j = j0 + jj;
                if (j >= n) break;
                const uint32_t sl = __shfl_sync(0xffffffffu, mine.x, j);
                const float wj = __shfl_sync(0xffffffffu, wmine, j);
                if (sl != cur) {
                    const bool open_start = seg_first && prev == cur;
                    if (open_start) acc.store(carry, D, lane);  // head: started in an earlier chunk, ends here
                    else acc.store(w.E + (size_t)cur * D, D, lane);
                    acc.clear();
                    cur = sl;
                    seg_first = false;
                }
#pragma unroll
                for (int i = 0; i < (VEC ? 4 * CPL : CPL); ++i) acc.v[i] = fmaf(wj, rowv[jj].v[i], acc.v[i]);
            }
        }
        tcur = __shfl_sync(0xffffffffu, tmine, n - 1);
    }
    const bool open_start = seg_first && prev == cur;
    const bool open_end = next == cur;
    if (open_end) acc.store(carry + D, D, lane);        // tail: continues in the next chunk
    else if (open_start) acc.store(carry, D, lane);     // head
    else acc.store(w.E + (size_t)cur * D, D, lane);
}

// The chunk in which a border-crossing segment starts adds up its pieces: its own tail, the tails of the chunks that the
// segment fills, the head in the chunk where it ends (the next row's start is the segment's end).  A warp adds a few
// pieces by itself; a popular row spans hundreds of chunks, and one warp would walk them one memory round trip after the
// other, so those are left to the whole CTA: 256 threads as 256 / (D / VEC) piece slots side by side, each with every
// slots-th piece, then the slots in order.  (One warp per row: 4 M lookups,
// D = 16, dE 187 us in chunks of 512 and 302 us in chunks of 128; now 142 and 121 us.)
#define DE_FIX_OWN 8    // pieces that a warp adds by itself
// No launch_dependents: the CTAs of the sweep that follows are placed when these are done.  Let in earlier, a grid of less than a
// wave went to the few SMs that had room by then and left the others idle.  Training calls, early / now, us: tables of 20 k rows: eight,
// 4x8x4, rank 32, 0.66 M lookups 818 / 677; one, 2x4x4, rank 32, 82 k lookups 264 / 223; one of four cores, rank 64, 447 / 421; larger
// grids lose the overlap of one launch: 8 tables, rank 16, 1.6 M lookups 588 / 591, 1 k lookups 103 / 104; four tables of 200 k
// rows, 4x4x4, rank 32, whose sweep is just a wave, 359 / 373 (neighbouring units on one SM share their slices).
template <bool VEC, int CPL>
__global__ void __launch_bounds__(256) k_dE_fix(WsView w)
{
    tt_pdl_wait();
    using piece_t = typename std::conditional<VEC, float4, float>::type;
    __shared__ piece_t s_part[256];
    __shared__ uint32_t s_chunk[8], s_slot[8], s_pieces[8];
    __shared__ uint32_t s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t chunk = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t U = w.counters[CTR_LEVEL0 + w.K];
    const uint32_t Ltot = w.cnt[U];
    const int64_t a64 = chunk << w.de_chunk_log, b64 = a64 + (1LL << w.de_chunk_log);
    const int D = w.D;
    if (b64 < Ltot) {
        const uint32_t last = w.chunk_slot[chunk + 1], from = tt_seg_start(w, last, U);   // the row after this chunk
        if (from < (uint32_t)b64 && from >= (uint32_t)a64) {                              // starts in it
            const uint32_t end = tt_seg_start(w, last + 1, U);
            const uint32_t pieces = ((end - 1u) >> w.de_chunk_log) - (uint32_t)chunk + 1u;
            if (pieces > DE_FIX_OWN) {
                if (lane == 0) {
                    const uint32_t i = atomicAdd(&s_n, 1u);
                    s_chunk[i] = (uint32_t)chunk;
                    s_slot[i] = last;
                    s_pieces[i] = pieces;
                }
            } else {
                RowAcc<VEC, CPL> acc;
                acc.clear();
#pragma unroll 4
                for (uint32_t i = 0; i + 1 < pieces; ++i) acc.add_row(w.carry + ((size_t)(chunk + i) * 2 + 1) * D, D, lane);
                acc.add_row(w.carry + (size_t)(chunk + pieces - 1) * 2 * D, D, lane);
                acc.store(w.E + (size_t)last * D, D, lane);
            }
        }
    }
    __syncthreads();
    const int cols = VEC ? D / 4 : D;                   // pieces of a row that the threads own
    const int width = cols < 256 ? cols : 256;
    const uint32_t slots = 256u / (uint32_t)width, slot = threadIdx.x / width;
    for (uint32_t q = 0; q < s_n; ++q) {
        const uint32_t pieces = s_pieces[q];
        const piece_t* src = reinterpret_cast<const piece_t*>(w.carry) + (size_t)s_chunk[q] * 2 * cols;
        for (int c0 = 0; c0 < cols; c0 += width) {
            const int c = c0 + threadIdx.x % width;
            RowAcc<VEC, 1> acc;                         // one piece of the row
            acc.clear();
            if (slot < slots && c < cols) {
#pragma unroll 8
                for (uint32_t i = slot; i < pieces; i += slots) {
                    const piece_t* x = src + ((size_t)i * 2 + (i + 1 < pieces ? 1 : 0)) * cols + c;
                    acc.add_row(reinterpret_cast<const float*>(x), VEC ? 4 : 1, 0);
                }
                acc.store(reinterpret_cast<float*>(&s_part[threadIdx.x]), VEC ? 4 : 1, 0);
            }
            __syncthreads();
            if (slot == 0 && c < cols) {
                acc.clear();
                for (uint32_t i = 0; i < slots; ++i)
                    acc.add_shared(&s_part[i * width + threadIdx.x]);
                acc.store(w.E + (size_t)s_slot[q] * D + (VEC ? 4 * c : c), VEC ? 4 : 1, 0);
            }
            __syncthreads();
        }
    }
}

// Fast variant for D/4 <= 32 float4 chunks per row: LPR lanes cover a row, 32/LPR rows per load instruction,
// NF load instructions issued back to back, then the rows are folded in position order.  Each sub-warp keeps
// its own partial sum; the sub-warps are combined only when a segment ends.  Segment starts inside a batch of
// 32 positions are found once with a ballot, so a window without a start costs 4 adds per load and nothing else.
template <int LPR, bool WT>
__global__ void __launch_bounds__(256, 5) k_dE_fast(WsView w, const float* __restrict__ grad_out)
{
    tt_pdl_enter();
    constexpr int RPI = 32 / LPR, NF = 4;
    const int lane = threadIdx.x & 31, sub = lane / LPR, lr = lane % LPR;
    const int64_t chunk = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    DePairs pairs(w, chunk);
    if (pairs.a >= pairs.b) return;
    pairs.begin<WT, false>(chunk, lane);
    const uint32_t a = pairs.a, b = pairs.b;
    if (a >= b) return;
    const int D = w.D, D4 = D >> 2;
    const bool lane_on = lr < D4;
    const uint32_t prev = pairs.prev, next = pairs.next_slot;
    const float4* __restrict__ G4 = reinterpret_cast<const float4*>(grad_out);
    float4* __restrict__ E4 = reinterpret_cast<float4*>(w.E);
    float4* carry4 = reinterpret_cast<float4*>(w.carry + (size_t)chunk * 2 * D);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t cur = pairs.s;
    bool seg_first = true;
    // close the running segment: combine the sub-warps, store (sub-warp 0 writes), clear
    auto close_segment = [&]() {
        float4* dst = (seg_first && prev == cur) ? carry4 : E4 + (size_t)cur * D4;   // head piece or whole segment
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        }
        if (sub == 0 && lane_on) dst[lr] = acc;
        acc = make_float4(0.f, 0.f, 0.f, 0.f);
        seg_first = false;
    };
    uint32_t last_slot = cur;  // slot of the position before the current batch
    for (uint32_t p0 = a; p0 < b; p0 += 32) {
        const int n = (int)min(32u, b - p0);
        const uint2 mine = make_uint2(pairs.rows(p0, n, lane), pairs.bag);
        const float wmine = pairs.factor;   // of this lane's pair
        if (p0 + 32 < b) pairs.fetch<WT>(p0 + 32, lane);
        // row index of this lane's pair inside grad_out viewed as [B*T][D]
        const uint32_t grow = lane < n ? mine.y * (uint32_t)w.T + (uint32_t)tt_find_table(w.tb[w.K], w.T, mine.x) : 0u;
        uint32_t before = __shfl_up_sync(0xffffffffu, mine.x, 1);
        if (lane == 0) before = last_slot;
        const unsigned starts = __ballot_sync(0xffffffffu, lane < n && mine.x != before);  // bit j: position j opens a segment
        last_slot = __shfl_sync(0xffffffffu, mine.x, n - 1);
        for (int j0 = 0; j0 < n; j0 += NF * RPI) {
            float4 v[NF];
#pragma unroll
            for (int jj = 0; jj < NF; ++jj) {
                const int j = j0 + jj * RPI + sub;
                const uint32_t gr = __shfl_sync(0xffffffffu, grow, j & 31);
                v[jj] = (j < n && lane_on) ? __ldg(G4 + (size_t)gr * D4 + lr) : make_float4(0.f, 0.f, 0.f, 0.f);
                if (WT) {
                    const float wj = __shfl_sync(0xffffffffu, wmine, j & 31);
                    v[jj].x *= wj; v[jj].y *= wj; v[jj].z *= wj; v[jj].w *= wj;
                }
            }
#pragma unroll
            for (int jj = 0; jj < NF; ++jj) {
                const int j = j0 + jj * RPI;
                if (((starts >> j) & ((1u << RPI) - 1u)) == 0u) {
                    acc.x += v[jj].x; acc.y += v[jj].y; acc.z += v[jj].z; acc.w += v[jj].w;
                } else {
#pragma unroll
                    for (int h = 0; h < RPI; ++h) {
                        if ((starts >> (j + h)) & 1u) {
                            close_segment();
                            cur = __shfl_sync(0xffffffffu, mine.x, (j + h) & 31);
                        }
                        if (sub == h) { acc.x += v[jj].x; acc.y += v[jj].y; acc.z += v[jj].z; acc.w += v[jj].w; }
                    }
                }
            }
        }
    }
    // last segment of the chunk
    {
        const bool open_start = seg_first && prev == cur;
        float4* dst = next == cur ? carry4 + D4 : (open_start ? carry4 : E4 + (size_t)cur * D4);  // tail / head / whole
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        }
        if (sub == 0 && lane_on) dst[lr] = acc;
    }
}

// The 32 grad_out rows of a batch of sorted positions are fetched into a per-warp buffer (8 KB with D = 64) with
// cp.async (all in flight at once, no staging registers), then every lane walks the batch in position
// order owning two of the 64 columns: one shared-memory load and two adds per row, a coalesced 256-byte store when a
// segment ends, and no shuffles to combine partial sums.  About half the instructions per lookup of k_dE_fast, which
// was bound by instruction issue.  Chunks, carries and the fix-up pass are those of k_dE / k_dE_fast.
#define DE_ODD_MOST 61   // with the up to three floats before it, a row fits sixteen pieces
#define DE_WARPS 7   // 4 CTAs x 7 warps x 8 KB of staging per SM
// DD = 128: rows of 512 bytes, two CTAs per SM (65 k lookups: dE with the pieces added up 38 -> 29 us against k_dE_fast).
// DD = 0: rows of any other length up to 61 floats.  A row starts anywhere in its first 16-byte piece; the pieces that it touches
// are staged as they lie (the last ones of grad_out cut to its end), and a lane picks columns lane and lane + 32 behind the row's
// shift.  1 M lookups of 45 floats: 112 -> 84 us against k_dE.
template <int DD, bool WT, bool JOIN>   // DD = D: 128 (four columns per lane), 64 (two), 32 (one), 16 (one, lanes 0..15) or 0
__global__ void __launch_bounds__(32 * DE_WARPS, DD == 128 ? 2 : 4) k_dE_stage(WsView w, const float* __restrict__ grad_out)
{
    if (JOIN) tt_pdl_wait(); else tt_pdl_enter();   // (the sweep comes next: see k_dE_fix)
    static_assert(DD == 128 || DD == 64 || DD == 32 || DD == 16 || DD == 0, "a lane owns DD / 32 columns (one column on the first DD lanes below 32)");
    constexpr bool ODD = DD == 0;
    constexpr int R4 = ODD ? 16 : DD / 4;         // float4 pieces per staged row
    constexpr int RPI = 32 / R4;                  // rows per cp.async instruction
    constexpr int VPL = ODD ? 2 : DD >= 32 ? DD / 32 : 1;   // columns per lane
    const int D = ODD ? w.D : DD;
    extern __shared__ __align__(16) float4 de_buf[];   // [DE_WARPS][32 rows][R4 float4]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, sub = lane / R4, lr = lane % R4;
    float4* buf = de_buf + (size_t)wid * 32 * R4;
    const float* bufv = reinterpret_cast<const float*>(buf);
    const int64_t chunk = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    DePairs pairs(w, chunk);
    if (pairs.a >= pairs.b) return;
    pairs.begin<WT, JOIN>(chunk, lane);
    const uint32_t a = pairs.a, b = pairs.b;
    if (a >= b) return;
    const uint32_t prev = pairs.prev, next = pairs.next_slot;
    const float4* __restrict__ G4 = reinterpret_cast<const float4*>(grad_out);
    float* carry = w.carry + (size_t)chunk * 2 * D;
    const uint32_t* __restrict__ tbK = w.tb[w.K];
    float acc[VPL], part[VPL];
#pragma unroll
    for (int x = 0; x < VPL; ++x) { acc[x] = 0.f; part[x] = 0.f; }
    uint32_t cur = pairs.s;
    bool seg_first = true;
    // slot range of the table the chunk is in: positions are sorted, so a batch rarely leaves it
    int tcur = tt_find_table(tbK, w.T, cur);
    uint32_t t_hi = tbK[tcur + 1];
    // two-level sum: rows are added into a per-batch partial (at most 32 terms) which is added to the segment's sum at
    // the end of the batch, so the rounding error of a long segment grows with sqrt(length / 32), not sqrt(length)
    auto store_row = [&](float* dst, bool with_part) {
        if (ODD) {
            if (lane < D) dst[lane] = acc[0] + (with_part ? part[0] : 0.f);
            if (lane + 32 < D) dst[lane + 32] = acc[VPL - 1] + (with_part ? part[VPL - 1] : 0.f);
        } else if (VPL == 4)
            reinterpret_cast<float4*>(dst)[lane] = make_float4(acc[0] + (with_part ? part[0] : 0.f), acc[1 % VPL] + (with_part ? part[1 % VPL] : 0.f),
                                                               acc[2 % VPL] + (with_part ? part[2 % VPL] : 0.f), acc[VPL - 1] + (with_part ? part[VPL - 1] : 0.f));
        else if (VPL == 2) reinterpret_cast<float2*>(dst)[lane] = make_float2(acc[0] + (with_part ? part[0] : 0.f), acc[VPL - 1] + (with_part ? part[VPL - 1] : 0.f));
        else if (lane < DD) dst[lane] = acc[0] + (with_part ? part[0] : 0.f);
    };
    auto close_segment = [&]() {
        store_row((seg_first && prev == cur) ? carry : w.E + (size_t)cur * D, true);   // head piece or whole segment
#pragma unroll
        for (int x = 0; x < VPL; ++x) { acc[x] = 0.f; part[x] = 0.f; }
        seg_first = false;
        ++cur;
    };
    for (uint32_t p0 = a; p0 < b; p0 += 32) {
        const int n = (int)min(32u, b - p0);
        unsigned starts;
        const bool plain = pairs.starts(p0, n, starts);
        const uint32_t row = plain ? cur + __popc(starts & (0xffffffffu >> (31 - lane))) : pairs.rows(p0, n, lane);
        const uint32_t bag = pairs.bag;
        const float wmine = pairs.factor;
        int tl = tcur;
        if (pairs.s >= t_hi) {
            tl = lane < n ? tt_find_table(tbK, w.T, row) : tcur;
            tcur = __shfl_sync(0xffffffffu, tl, n - 1);
            t_hi = tbK[tcur + 1];
        }
        const uint32_t grow = bag * (uint32_t)w.T + (uint32_t)tl;   // row of grad_out viewed as [B*T][DD]
        const uint32_t shift = (grow * (uint32_t)D) & 3u;   // (ODD) floats before the row in its first piece
        if constexpr (ODD) {
            const uint64_t all = (uint64_t)w.B * w.T * D;
#pragma unroll 4
            for (int jj = 0; jj < 32 / RPI; ++jj) {
                if (RPI * jj >= n) break;
                const int j = RPI * jj + sub;
                const uint64_t start = (uint64_t)__shfl_sync(0xffffffffu, grow, j) * (uint32_t)D, at = (start & ~(uint64_t)3) + 4 * lr;
                if (j < n && at < start + D) tt_cp_async16_cut(buf + j * R4 + lr, grad_out + at, all - at);
            }
        } else if (n == 32) {   // all windows of a chunk but its last: no per-row test
#pragma unroll
            for (int jj = 0; jj < 32 / RPI; ++jj) {
                const int j = RPI * jj + sub;
                const uint32_t gr = __shfl_sync(0xffffffffu, grow, j);
                tt_cp_async16(buf + j * R4 + lr, G4 + (size_t)gr * R4 + lr);
            }
        } else {
#pragma unroll
            for (int jj = 0; jj < 32 / RPI; ++jj) {
                const int j = RPI * jj + sub;
                const uint32_t gr = __shfl_sync(0xffffffffu, grow, j);
                if (j < n) tt_cp_async16(buf + j * R4 + lr, G4 + (size_t)gr * R4 + lr);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (p0 + 32 < b) pairs.fetch<WT>(p0 + 32, lane);   // the next batch's arrive while the rows are in flight
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        auto add_row = [&](int j) {
            float x[VPL];
            if (ODD) {
                const float* src = bufv + j * 64 + __shfl_sync(0xffffffffu, shift, j) + lane;
                x[0] = lane < D ? src[0] : 0.f;
                x[VPL - 1] = lane + 32 < D ? src[32] : 0.f;
            } else if (VPL == 4) {
                const float4 v = buf[j * 32 + lane];
                x[0] = v.x; x[1 % VPL] = v.y; x[2 % VPL] = v.z; x[VPL - 1] = v.w;
            } else if (VPL == 2) {
                const float2 v = reinterpret_cast<const float2*>(bufv)[j * 32 + lane];
                x[0] = v.x; x[VPL - 1] = v.y;
            } else x[0] = bufv[j * DD + (lane & (DD - 1))];
            if (WT) {
                const float wj = __shfl_sync(0xffffffffu, wmine, j);
#pragma unroll
                for (int c = 0; c < VPL; ++c) x[c] *= wj;
            }
#pragma unroll
            for (int c = 0; c < VPL; ++c) part[c] += x[c];
        };
        // eight rows at a time; a run of eight without a segment start (popular rows: most lookups sit in segments far
        // longer than a batch) is added without looking at the start bits
        for (int j0 = 0; plain && j0 < n; j0 += 8) {
            if (j0 + 8 <= n && ((starts >> j0) & 0xffu) == 0u) {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) add_row(j0 + jj);
            } else if (j0 + 8 <= n && ((starts >> j0) & 0xffu) == 0xffu) {
                // eight starts in a row (rows looked up once: most distinct rows): the first closes the running segment,
                // the next seven rows are whole segments of one row each and are copied out, the eighth opens a new one
                close_segment();
                float* dst = w.E + (size_t)cur * D;
                cur += 7;
#pragma unroll
                for (int jj = 0; jj < 7; ++jj, dst += D) {
                    add_row(j0 + jj);
                    if (ODD) {
                        if (lane < D) dst[lane] = part[0];
                        if (lane + 32 < D) dst[lane + 32] = part[VPL - 1];
                    } else if (VPL == 4) reinterpret_cast<float4*>(dst)[lane] = make_float4(part[0], part[1 % VPL], part[2 % VPL], part[VPL - 1]);
                    else if (VPL == 2) reinterpret_cast<float2*>(dst)[lane] = make_float2(part[0], part[VPL - 1]);
                    else if (lane < DD) dst[lane] = part[0];
#pragma unroll
                    for (int c = 0; c < VPL; ++c) part[c] = 0.f;
                }
                add_row(j0 + 7);
            } else if (VPL == 4 && j0 + 8 <= n) {
                // segments of a few rows: with fourteen warps per SM the eight rows are fetched before the first start is looked at (0.66 M
                // lookups in eight tables of 20 k rows, 4 M in four of 200 k, one of 200 k 1.5 M, us: dE 59 / 50, 269 / 228, 103 / 87;
                // k_dE_fast 47, 218, 87, and 701 against 535 with 12 M in four)
                float4 v[8];
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) {
                    v[jj] = buf[(j0 + jj) * R4 + lr];
                    if (WT) {
                        const float wj = __shfl_sync(0xffffffffu, wmine, j0 + jj);
                        v[jj] = make_float4(v[jj].x * wj, v[jj].y * wj, v[jj].z * wj, v[jj].w * wj);
                    }
                }
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) {
                    if ((starts >> (j0 + jj)) & 1u) close_segment();
                    part[0] += v[jj].x; part[1 % VPL] += v[jj].y; part[2 % VPL] += v[jj].z; part[VPL - 1] += v[jj].w;
                }
            } else {
                const int j1 = min(j0 + 8, n);
                for (int j = j0; j < j1; ++j) {
                    if ((starts >> j) & 1u) close_segment();
                    add_row(j);
                }
            }
        }
        if (!plain)
            for (int j = 0; j < n; ++j) {
                const uint32_t rj = __shfl_sync(0xffffffffu, row, j);
                if (rj != cur) {
                    close_segment();
                    cur = rj;
                }
                add_row(j);
            }
#pragma unroll
        for (int c = 0; c < VPL; ++c) { acc[c] += part[c]; part[c] = 0.f; }
        __syncwarp();
    }
    {   // last segment of the chunk: tail / head / whole
        const bool open_start = seg_first && prev == cur;
        store_row(next == cur ? carry + D : (open_start ? carry : w.E + (size_t)cur * D), false);
    }
    if (JOIN) de_finish<!ODD>(w, pairs, chunk, cur, lane);
}

template <bool WT, bool JOIN>
static auto de_stage_kernel(int D) -> void (*)(WsView, const float*)
{
    return D == 0 ? k_dE_stage<0, WT, JOIN> : D == 128 ? k_dE_stage<128, WT, JOIN> : D == 64 ? k_dE_stage<64, WT, JOIN>
         : D == 32 ? k_dE_stage<32, WT, JOIN> : k_dE_stage<16, WT, JOIN>;
}

template <bool VEC, int CPL>
static cudaError_t launch_dE_t(tt_emb* h, const float* grad_out, cudaStream_t s)
{
    const int64_t chunks = (h->v.L + (1LL << h->v.de_chunk_log) - 1) >> h->v.de_chunk_log;
    const int grid = (int)((chunks + 7) / 8);
    if (grid > 0) {
        const int D4 = h->D / 4;
        const bool wt = tt_weighted(h->v);
        const bool join = chunks <= (h->D > 32 ? 2 * DE_JOIN_CHUNKS : DE_JOIN_CHUNKS);
        const bool odd = !VEC && h->D <= DE_ODD_MOST && (reinterpret_cast<uintptr_t>(grad_out) & 15) == 0;
        if (odd || (VEC && (h->D == 128 || h->D == 64 || h->D == 32 || h->D == 16))) {
            const size_t smem = (size_t)DE_WARPS * 32 * (odd ? 16 : h->D / 4) * sizeof(float4);
            auto kern = join ? (wt ? de_stage_kernel<true, true>(odd ? 0 : h->D) : de_stage_kernel<false, true>(odd ? 0 : h->D))
                             : (wt ? de_stage_kernel<true, false>(odd ? 0 : h->D) : de_stage_kernel<false, false>(odd ? 0 : h->D));
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            const int sgrid = (int)((chunks + DE_WARPS - 1) / DE_WARPS);
            if ((e = tt_launch_pdl(kern, dim3(sgrid), dim3(32 * DE_WARPS), smem, s, h->v, grad_out)) != cudaSuccess) return e;
            tt_note_launch();
            if (join) return cudaGetLastError();
        } else
        if (VEC && D4 <= 8) { if (wt) k_dE_fast<8, true><<<grid, 256, 0, s>>>(h->v, grad_out); else k_dE_fast<8, false><<<grid, 256, 0, s>>>(h->v, grad_out); tt_note_launch(); }
        else if (VEC && D4 <= 16) { if (wt) k_dE_fast<16, true><<<grid, 256, 0, s>>>(h->v, grad_out); else k_dE_fast<16, false><<<grid, 256, 0, s>>>(h->v, grad_out); tt_note_launch(); }
        else if (VEC && D4 <= 32) { if (wt) k_dE_fast<32, true><<<grid, 256, 0, s>>>(h->v, grad_out); else k_dE_fast<32, false><<<grid, 256, 0, s>>>(h->v, grad_out); tt_note_launch(); }
        else { k_dE<VEC, CPL><<<grid, 256, 0, s>>>(h->v, grad_out); tt_note_launch(); }
        cudaError_t ef = tt_launch_pdl(k_dE_fix<VEC, CPL>, dim3(grid), dim3(256), 0, s, h->v);
        if (ef != cudaSuccess) return ef;
        tt_note_launch();
    }
    return cudaGetLastError();
}

cudaError_t tt_launch_bwd_dE(tt_emb* h, const float* grad_out, cudaStream_t s)
{
    const int D = h->D;
    const bool vec = (D % 4 == 0) && ((reinterpret_cast<uintptr_t>(grad_out) & 15) == 0);
    if (vec) {
        if (D <= 128) return launch_dE_t<true, 1>(h, grad_out, s);
        if (D <= 256) return launch_dE_t<true, 2>(h, grad_out, s);
        if (D <= 512) return launch_dE_t<true, 4>(h, grad_out, s);
        return launch_dE_t<true, 8>(h, grad_out, s);
    }
    if (D <= 32) return launch_dE_t<false, 1>(h, grad_out, s);
    if (D <= 64) return launch_dE_t<false, 2>(h, grad_out, s);
    if (D <= 128) return launch_dE_t<false, 4>(h, grad_out, s);
    if (D <= 256) return launch_dE_t<false, 8>(h, grad_out, s);
    if (D <= 512) return launch_dE_t<false, 16>(h, grad_out, s);
    return launch_dE_t<false, 32>(h, grad_out, s);
}

// ---------------------------------------------------------------------------------------------- 3. last level

// dC of the batch's groups to the level above (K = 2: it is the gradient of the first core's slice itself); ends with a barrier
template <int THREADS>
__device__ __forceinline__ void gen_hand_up(const WsView& w, const TableDesc& td, int cnt, const GenBatch& b, const float* dCs)
{
    const int K = w.K, Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb);
    for (int it = threadIdx.x; it < cnt * Pm * rb; it += THREADS) {
        const int q = it / (Pm * rb), e = it - q * (Pm * rb), p = e / rb;
        float* dst = K >= 3 ? w.dP[K - 1] + (size_t)b.g[q] * w.stride[K - 1] : td.grad[0] + (size_t)b.val[q] * td.slice_floats[0];
        const float x = dCs[q * (Pm * pitch) + p * pitch + (e - p * rb)];
        if (b.part[q]) atomicAdd(dst + e, x);   // K = 2: the first core's gradient starts at zero
        else dst[e] = x;
    }
    __syncthreads();
}

// any shape: batches of groups spread flat over the CTA (generic.cuh)
__global__ void __launch_bounds__(GEN_THREADS, 3) k_sweep_bwd_any(WsView w, int vbase)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ GenBatch b;
    __shared__ float4 s_part[GEN_THREADS];
    const int t = w.vlist[vbase + blockIdx.y], K = w.K;
    const uint2 rng = w.unit_rng[t * w.units_per_table + blockIdx.x];
    const TableDesc& td = w.tdesc[t];
    const int stripe = (blockIdx.x + blockIdx.y) % TT_STRIPES;
    float* gk = w.gpart + (size_t)stripe * w.gpart_stride + td.gpart_off;
    float *Cs = sm, *dCs = sm + GEN_C_FLOATS;
    const bool vec = (td.d[K - 1] & 3) == 0;
    const int Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb);
    const uint32_t ng = (uint32_t)gen_groups(td, K);
    uint2 groups, range;
    gen_unit(w, t, rng, groups, range);
    for (uint32_t base = groups.x; base < groups.y; base += ng) {
        const int cnt = (int)min(ng, groups.y - base);
        for (int i = threadIdx.x; i < cnt * Pm * pitch; i += GEN_THREADS) dCs[i] = 0.f;
        gen_batch_begin(w, td, base, cnt, range, b);
        gen_batch_c<GEN_THREADS>(w, td, cnt, b, Cs);
        const uint32_t rows = b.row0[cnt];
        for (uint32_t r0 = 0; r0 < rows; r0 += GEN_ROWS) {
            const int n = (int)min((uint32_t)GEN_ROWS, rows - r0);
            gen_rows(w, td, cnt, r0, n, b);
            if (vec) {
                gen_backward_slice<true>(w, td, n, b, Cs, gk);
                gen_backward_dc<true>(w, td, r0, n, b, dCs, s_part);
            } else {
                gen_backward_slice<false>(w, td, n, b, Cs, gk);
                gen_backward_dc<false>(w, td, r0, n, b, dCs, s_part);
            }
            __syncthreads();
        }
        gen_hand_up<GEN_THREADS>(w, td, cnt, b, dCs);
    }
}

// the same for one last dim factor of 1, 2, 3, 5, 6 or 7
template <int DK>
__global__ void __launch_bounds__(GEN_ODD_THREADS, 6) k_sweep_bwd_odd(WsView w, int vbase, int c_floats)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ GenBatch b;
    __shared__ float s_part[4 * GEN_P * GEN_ODD_THREADS];
    const int t = w.vlist[vbase + blockIdx.y], K = w.K;
    const uint2 rng = w.unit_rng[t * w.units_per_table + blockIdx.x];
    const TableDesc& td = w.tdesc[t];
    const int stripe = (blockIdx.x + blockIdx.y) % TT_STRIPES;
    float* gk = w.gpart + (size_t)stripe * w.gpart_stride + td.gpart_off;
    float *Cs = sm, *dCs = sm + c_floats, *Es = dCs + c_floats;
    const int Pm = td.P[K - 1], rb = td.r[K - 1], pitch = gen_pitch(rb);
    const uint32_t ng = (uint32_t)gen_groups(td, K), chunk = (uint32_t)gen_stage_rows(w.D);
    uint2 groups, range;
    gen_unit(w, t, rng, groups, range);
    for (uint32_t base = groups.x; base < groups.y; base += ng) {
        const int cnt = (int)min(ng, groups.y - base);
        for (int i = threadIdx.x; i < cnt * Pm * pitch; i += GEN_ODD_THREADS) dCs[i] = 0.f;
        gen_batch_begin(w, td, base, cnt, range, b);
        gen_batch_c<GEN_ODD_THREADS>(w, td, cnt, b, Cs);
        const uint32_t rows = b.row0[cnt];
        for (uint32_t r0 = 0; r0 < rows; r0 += chunk) {
            const int n = (int)min(chunk, rows - r0);
            gen_rows(w, td, cnt, r0, n, b);
            gen_stage(w, n, b, Es);
            gen_slice_odd<DK>(w, td, n, b, Cs, Es, gk);
            gen_dc_odd<DK>(w, td, r0, n, b, Es, dCs, s_part);
            __syncthreads();
        }
        gen_hand_up<GEN_ODD_THREADS>(w, td, cnt, b, dCs);
    }
}

// ---- register-tiled backward of the last two levels (same shape variants as the forward sweep) ----------------
//
// One warp per group.  C is rebuilt in shared memory, then two passes over the group's rows:
//   pass A  dC[p][b] += sum_j dE_u[p][j] * D_u[b][j]: a lane owns TP rows p for all b (TP*RB accumulators) and
//           one of 32*TP/PM concurrent rows; D streams as float4 (16 FMAs per load at TP = 4).  The row-slots
//           are then combined by a reduce-scatter of warp shuffles and each lane writes its share of dC (Eq. 2:
//           the sum over the rows sharing C is formed before anything moves up a level).
//   pass B  dG_K[i_K][b][j] += sum_p C[p][b] * dE_u[p][j]: a lane owns RB*TP/PM values of b for all p
//           (PM*RB*TP/PM registers of C) and streams the float4 rows of dE (8*TP FMAs per load at PM = 16).
//           The lane's 4*RB*TP/PM results are contiguous in the slice and go out as vector reductions.

__device__ __forceinline__ void tt_red_v4(float* p, float x, float y, float z, float wv)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(wv) : "memory");
}

// RBP > 0: C is stored as [P][RBP + 8] (rows of r_{K-1} = RBP values, stride RBP + 8 floats), the layout whose transposed
// fragment loads in the tensor-core dG pass are free of bank conflicts; RBP = 0: plain [M][cols].
template <int M, int CPL, int RBP = 0>
__device__ __forceinline__ void tt_warp_mid_b(const float* As, const float* __restrict__ Bsl, float* Cs, int ra, int cols, int lane)
{
    const int c4n = cols >> 2;
    const int LA = (c4n / CPL) < 32 ? (c4n / CPL) : 32;
    const int NS = 32 / LA;
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
            for (int m = 0; m < M; ++m) {
                const int col = 4 * (ll + i * LA);
                float* dst = RBP > 0 ? Cs + (m * (cols / (RBP > 0 ? RBP : 1)) + col / (RBP > 0 ? RBP : 1)) * (RBP + 8) + col % (RBP > 0 ? RBP : 1)
                                     : Cs + m * cols + col;
                *reinterpret_cast<float4*>(dst) = make_float4(acc[i][m][0], acc[i][m][1], acc[i][m][2], acc[i][m][3]);
            }
    }
}

template <int PM, int RB_, int TP>
__device__ __forceinline__ void tt_warp_rows_dC(const WsView& w, const TableDesc& td, uint32_t u0, uint32_t u1, uint32_t row_base,
                                                float* dPdst, int lane)
{
    constexpr int LR = PM / TP, RW = 32 / LR, NV = TP * RB_;
    const int q = lane % LR, slot = lane / LR;
    const int K = w.K;
    const float* __restrict__ GK = td.core[K - 1];
    const uint32_t* __restrict__ rows = w.val[K];
    const float4* __restrict__ E4 = reinterpret_cast<const float4*>(w.E);
    float dc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) dc[i] = 0.f;
    for (uint32_t ub = u0; ub < u1; ub += RW) {
        const uint32_t u = ub + slot;
        const bool act = u < u1;
        const uint32_t iK = act ? rows[u] - row_base : 0u;
        const float4* __restrict__ D4 = reinterpret_cast<const float4*>(GK + (size_t)iK * (RB_ * 4));
        float4 e[TP];
#pragma unroll
        for (int i = 0; i < TP; ++i) e[i] = act ? __ldg(E4 + (size_t)u * PM + TP * q + i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int b = 0; b < RB_; ++b) {
            const float4 d = __ldg(D4 + b);
#pragma unroll
            for (int i = 0; i < TP; ++i) {
                float a = dc[i * RB_ + b];
                a = fmaf(e[i].x, d.x, a); a = fmaf(e[i].y, d.y, a); a = fmaf(e[i].z, d.z, a); a = fmaf(e[i].w, d.w, a);
                dc[i * RB_ + b] = a;
            }
        }
    }
    // reduce-scatter over the RW row-slots: after the step with lane bit o, a lane keeps the half selected by that bit
    int base = 0;
    int n = NV;
#pragma unroll
    for (int o = 16; o >= LR; o >>= 1) {
        n >>= 1;
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < NV / 2; ++i) {
            if (i < n) {
                const float send = hi ? dc[i] : dc[i + n];
                const float recv = __shfl_xor_sync(0xffffffffu, send, o);
                dc[i] = (hi ? dc[i + n] : dc[i]) + recv;
            }
        }
        base += hi ? n : 0;
    }
    // the lane now holds dc[0..n) = dC values [base, base+n) of its TP rows (value v <-> row v / RB_, column v % RB_)
    constexpr int NF = NV / RW;
    float* dst = dPdst + (TP * q + base / RB_) * RB_ + base % RB_;
    if constexpr (NF >= 4) {
#pragma unroll
        for (int i = 0; i < NF / 4; ++i)
            *reinterpret_cast<float4*>(dst + 4 * i) = make_float4(dc[4 * i], dc[4 * i + 1], dc[4 * i + 2], dc[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < NF; ++i) dst[i] = dc[i];
    }
}

template <int PM, int RB_, int TP>
__device__ __forceinline__ void tt_warp_rows_dG(const float* Cs, const WsView& w, uint32_t u0, uint32_t u1, uint32_t row_base,
                                                float* gk, int lane)
{
    constexpr int LR = PM / TP, RW = 32 / LR, BQ = RB_ / LR;
    const int q = lane % LR, slot = lane / LR;
    const uint32_t* __restrict__ rows = w.val[w.K];
    const float4* __restrict__ E4 = reinterpret_cast<const float4*>(w.E);
    float c2[PM][BQ];
#pragma unroll
    for (int p = 0; p < PM; ++p)
#pragma unroll
        for (int bi = 0; bi < BQ; ++bi) c2[p][bi] = Cs[p * RB_ + BQ * q + bi];
    for (uint32_t ub = u0; ub < u1; ub += RW) {
        const uint32_t u = ub + slot;
        const bool act = u < u1;
        const uint32_t ur = act ? u : u0;
        float4 acc[BQ];
#pragma unroll
        for (int bi = 0; bi < BQ; ++bi) acc[bi] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int p = 0; p < PM; ++p) {
            const float4 e = __ldg(E4 + (size_t)ur * PM + p);
#pragma unroll
            for (int bi = 0; bi < BQ; ++bi) {
                acc[bi].x = fmaf(c2[p][bi], e.x, acc[bi].x);
                acc[bi].y = fmaf(c2[p][bi], e.y, acc[bi].y);
                acc[bi].z = fmaf(c2[p][bi], e.z, acc[bi].z);
                acc[bi].w = fmaf(c2[p][bi], e.w, acc[bi].w);
            }
        }
        if (act) {
            const uint32_t iK = rows[u] - row_base;
            float* dst = gk + (size_t)iK * (RB_ * 4) + (BQ * q) * 4;
#pragma unroll
            for (int bi = 0; bi < BQ; ++bi) tt_red_v4(dst + 4 * bi, acc[bi].x, acc[bi].y, acc[bi].z, acc[bi].w);
        }
    }
}

// ---- tensor-core (3xTF32, m16n8k8) forms of the two row passes, d_K = 4 ---------------------------------------
//
// pass A  dC[p][b] = sum over the group's rows u and j of dE_u[p][j] * D_u[b][j]:  M = 16 rows p, N = 8 values of b,
//         K = 8 = two rows x 4 columns j.  The sum over the rows that share C (Eq. 2) is the accumulation over
//         k-steps, so dC ends up complete in the accumulator fragments (PM*RB/32 registers) and is written once:
//         no cross-lane reduction at all.
// pass B  dG_K[i_K(u)][b][j] += sum_p C[p][b] * dE_u[p][j]:  M = 16 values of b, K = 8 rows p, N = 8 = two rows x 4
//         columns j; C^T fragments are fixed per group.  Results leave as 8-byte vector reductions.
__device__ __forceinline__ void tt_red_v2(float* p, float x, float y)
{
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x), "f"(y) : "memory");
}

template <int PM, int RB_>
__device__ __forceinline__ void tt_warp_rows_dC_mma(const WsView& w, const TableDesc& td, uint32_t u0, uint32_t u1, uint32_t row_base,
                                                    float* dPdst, int lane)
{
    static_assert(PM % 16 == 0, "whole row tiles");
    constexpr int MT = PM / 16, NT = RB_ / 8;
    const int g = lane >> 2, t = lane & 3;
    const int K = w.K;
    const float* __restrict__ GK = td.core[K - 1];
    const uint32_t* __restrict__ rows = w.val[K];
    // acc: tensor-core accumulators, folded into tot (rounded fp32 adds) every sixteen row pairs: the tensor core adds
    // with truncation, so a long chain (a group can have hundreds of rows) would drift by chain length * 2^-24
    float acc[MT][NT][4], tot[MT][NT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int x = 0; x < 4; ++x) { acc[mt][nt][x] = 0.f; tot[mt][nt][x] = 0.f; }
    for (uint32_t ub0 = u0; ub0 < u1; ub0 += 32) {
    const uint32_t ub1 = min(ub0 + 32u, u1);
#pragma unroll 2
    for (uint32_t ub = ub0; ub < ub1; ub += 2) {
        const bool two = ub + 1 < u1;
        const uint32_t ua = ub, uc = two ? ub + 1 : ub;
        const float* __restrict__ Ea = w.E + (size_t)ua * (PM * 4) + t;
        const float* __restrict__ Ec = w.E + (size_t)uc * (PM * 4) + t;
        const float* __restrict__ Da = GK + (size_t)(rows[ua] - row_base) * (RB_ * 4) + t;
        const float* __restrict__ Dc = GK + (size_t)(rows[uc] - row_base) * (RB_ * 4) + t;
        Tf32Pair a[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            a[mt][0] = tt_split_tf32(__ldg(Ea + (16 * mt + g) * 4));
            a[mt][1] = tt_split_tf32(__ldg(Ea + (16 * mt + g + 8) * 4));
            a[mt][2] = tt_split_tf32(two ? __ldg(Ec + (16 * mt + g) * 4) : 0.f);
            a[mt][3] = tt_split_tf32(two ? __ldg(Ec + (16 * mt + g + 8) * 4) : 0.f);
        }
        float bv[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            bv[nt][0] = __ldg(Da + (8 * nt + g) * 4);
            bv[nt][1] = __ldg(Dc + (8 * nt + g) * 4);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            Tf32Pair b[2];
            b[0] = tt_split_tf32(bv[nt][0]);
            b[1] = tt_split_tf32(bv[nt][1]);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) tt_mma_3xtf32(acc[mt][nt], a[mt], b);
        }
    }
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int x = 0; x < 4; ++x) { tot[mt][nt][x] += acc[mt][nt][x]; acc[mt][nt][x] = 0.f; }
    }
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            *reinterpret_cast<float2*>(dPdst + (16 * mt + g) * RB_ + 8 * nt + 2 * t) = make_float2(tot[mt][nt][0], tot[mt][nt][1]);
            *reinterpret_cast<float2*>(dPdst + (16 * mt + g + 8) * RB_ + 8 * nt + 2 * t) = make_float2(tot[mt][nt][2], tot[mt][nt][3]);
        }
}

template <int PM, int RB_>
__device__ __forceinline__ void tt_warp_rows_dG_mma(const float* Cs, const WsView& w, uint32_t u0, uint32_t u1, uint32_t row_base,
                                                    float* gk, int lane)
{
    constexpr int MT = RB_ / 16, KT = PM / 8;
    const int g = lane >> 2, t = lane & 3;
    const uint32_t* __restrict__ rows = w.val[w.K];
    Tf32Pair a[MT][KT][4];   // A[m = b][k = p] = C[p][b]
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int kt = 0; kt < KT; ++kt) {
            a[mt][kt][0] = tt_split_tf32(Cs[(8 * kt + t) * (RB_ + 8) + 16 * mt + g]);
            a[mt][kt][1] = tt_split_tf32(Cs[(8 * kt + t) * (RB_ + 8) + 16 * mt + g + 8]);
            a[mt][kt][2] = tt_split_tf32(Cs[(8 * kt + t + 4) * (RB_ + 8) + 16 * mt + g]);
            a[mt][kt][3] = tt_split_tf32(Cs[(8 * kt + t + 4) * (RB_ + 8) + 16 * mt + g + 8]);
        }
    const int rb_ = g >> 2, jb = g & 3;       // B fragment: row rb_ of the pair, column jb of dE
    const int rc = t >> 1, jc = 2 * (t & 1);  // C fragment: row rc of the pair, columns jc, jc+1
#pragma unroll 2
    for (uint32_t ub = u0; ub < u1; ub += 2) {
        const uint32_t ul = min(ub + (uint32_t)rb_, u1 - 1);
        const bool valid = ub + (uint32_t)rb_ < u1;
        const float* __restrict__ El = w.E + (size_t)ul * (PM * 4) + jb;
        float acc[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) { acc[mt][0] = 0.f; acc[mt][1] = 0.f; acc[mt][2] = 0.f; acc[mt][3] = 0.f; }
        float bv[KT][2];
#pragma unroll
        for (int kt = 0; kt < KT; ++kt) {
            bv[kt][0] = valid ? __ldg(El + (8 * kt + t) * 4) : 0.f;
            bv[kt][1] = valid ? __ldg(El + (8 * kt + t + 4) * 4) : 0.f;
        }
#pragma unroll
        for (int kt = 0; kt < KT; ++kt) {
            Tf32Pair b[2];
            b[0] = tt_split_tf32(bv[kt][0]);
            b[1] = tt_split_tf32(bv[kt][1]);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) tt_mma_3xtf32(acc[mt], a[mt][kt], b);
        }
        const uint32_t us = ub + (uint32_t)rc;
        if (us < u1) {
            float* dst = gk + (size_t)(rows[us] - row_base) * (RB_ * 4) + jc;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                tt_red_v2(dst + (16 * mt + g) * 4, acc[mt][0], acc[mt][1]);
                tt_red_v2(dst + (16 * mt + g + 8) * 4, acc[mt][2], acc[mt][3]);
            }
        }
    }
}

// Both row passes in one loop over the group's row pairs, for C of 8 rows: the row ids and the dE rows come from memory once (the
// second fragment layout of dE is served by L1), dC accumulates across the loop, dG_K tiles leave per pair.  C of 8 rows would fill half
// of the row tiles of dC, so that product runs transposed, dC^T[b][p] += sum_{(row, j)} D_row[b][j] * dE_row[p][j], M = b, N = 8
// columns p, K = 8 = two rows x 4 columns j.
template <int RB_, int CS>   // CS: row stride of C in shared memory
__device__ __forceinline__ void tt_warp_rows_bwd_mma(const float* Cs, const WsView& w, const TableDesc& td, uint32_t u0, uint32_t u1,
                                                     uint32_t row_base, float* dPdst, float* gk, int lane)
{
    constexpr int PM = 8, MT = RB_ / 16, NT = RB_ / 8;
    const int g = lane >> 2, t = lane & 3;
    const int K = w.K;
    const float* __restrict__ GK = td.core[K - 1];
    const uint32_t* __restrict__ rows = w.val[K];
    Tf32Pair ct[MT][4];         // A[m = b][k = p] = C[p][b]
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        ct[mt][0] = tt_split_tf32(Cs[t * CS + 16 * mt + g]);
        ct[mt][1] = tt_split_tf32(Cs[t * CS + 16 * mt + g + 8]);
        ct[mt][2] = tt_split_tf32(Cs[(t + 4) * CS + 16 * mt + g]);
        ct[mt][3] = tt_split_tf32(Cs[(t + 4) * CS + 16 * mt + g + 8]);
    }
    float dc[MT][4], dct[MT][4];   // tensor-core accumulators and their rounded running sums (see tt_warp_rows_dC_mma)
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int x = 0; x < 4; ++x) { dc[mt][x] = 0.f; dct[mt][x] = 0.f; }
    const int rb_ = g >> 2, jb = g & 3;       // dG B fragment: row rb_ of the pair, column jb of dE
    const int rc = t >> 1, jc = 2 * (t & 1);  // dG C fragment: row rc of the pair, columns jc, jc+1
    for (uint32_t ub0 = u0; ub0 < u1; ub0 += 32) {
    const uint32_t ub1 = min(ub0 + 32u, u1);
    // last digits of the 32 rows, one per lane (a load per pair put two dependent loads before every product: 240-table workload,
    // sweep 4.47 -> 4.16 ms)
    const uint32_t ids = ub0 + lane < u1 ? rows[ub0 + lane] - row_base : 0u;
    for (uint32_t ub = ub0; ub < ub1; ub += 2) {
        const bool two = ub + 1 < u1;
        const uint32_t ua = ub, uc = two ? ub + 1 : ub;
        const uint32_t iKa = __shfl_sync(0xffffffffu, ids, ua - ub0), iKc = __shfl_sync(0xffffffffu, ids, uc - ub0);
        const float* __restrict__ Ea = w.E + (size_t)ua * (PM * 4);
        const float* __restrict__ Ec = w.E + (size_t)uc * (PM * 4);
        // ---- loads: dE as B fragment (dC), slices as A fragments (dC), dE as B fragment (dG)
        const float e0 = __ldg(Ea + g * 4 + t), e1 = two ? __ldg(Ec + g * 4 + t) : 0.f;   // dE_a[p = g][j = t], dE_c[g][t]
        const float* __restrict__ Da = GK + (size_t)iKa * (RB_ * 4) + t;
        const float* __restrict__ Dc = GK + (size_t)iKc * (RB_ * 4) + t;
        float dv[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            // (dv[2 mt][.], dv[2 mt + 1][.] are the A fragment rows b = 16 mt + g and + 8 of D_a, D_c)
            dv[nt][0] = __ldg(Da + (8 * nt + g) * 4);
            dv[nt][1] = two ? __ldg(Dc + (8 * nt + g) * 4) : 0.f;
        }
        const bool valid = rb_ == 0 || two;
        const float* __restrict__ El = (rb_ == 0 ? Ea : Ec) + jb;
        const float v0 = valid ? __ldg(El + t * 4) : 0.f, v1 = valid ? __ldg(El + (t + 4) * 4) : 0.f;
        // ---- dC += dE . D^T
        {
            const Tf32Pair b[2] = {tt_split_tf32(e0), tt_split_tf32(e1)};
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                const Tf32Pair a[4] = {tt_split_tf32(dv[2 * mt][0]), tt_split_tf32(dv[2 * mt + 1][0]), tt_split_tf32(dv[2 * mt][1]), tt_split_tf32(dv[2 * mt + 1][1])};
                tt_mma_3xtf32(dc[mt], a, b);
            }
        }
        // ---- dG_K[i_K] += C^T . dE
        {
            const Tf32Pair b[2] = {tt_split_tf32(v0), tt_split_tf32(v1)};
            float acc[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                acc[mt][0] = 0.f; acc[mt][1] = 0.f; acc[mt][2] = 0.f; acc[mt][3] = 0.f;
                tt_mma_3xtf32(acc[mt], ct[mt], b);
            }
            if (rc == 0 || two) {
                float* dst = gk + (size_t)(rc == 0 ? iKa : iKc) * (RB_ * 4) + jc;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    tt_red_v2(dst + (16 * mt + g) * 4, acc[mt][0], acc[mt][1]);
                    tt_red_v2(dst + (16 * mt + g + 8) * 4, acc[mt][2], acc[mt][3]);
                }
            }
        }
    }
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int x = 0; x < 4; ++x) { dct[mt][x] += dc[mt][x]; dc[mt][x] = 0.f; }
    }
    // the lane holds dC[p = 2t][b], dC[2t + 1][b] for b = 16 mt + g and b + 8
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        dPdst[(2 * t) * RB_ + 16 * mt + g] = dct[mt][0];
        dPdst[(2 * t + 1) * RB_ + 16 * mt + g] = dct[mt][1];
        dPdst[(2 * t) * RB_ + 16 * mt + g + 8] = dct[mt][2];
        dPdst[(2 * t + 1) * RB_ + 16 * mt + g + 8] = dct[mt][3];
    }
}

template <int PM, int RB_, int TP, int M, int CPL, bool MMA>
__device__ __forceinline__ void tt_sweep_bwd_fast(const WsView& w, const TableDesc& td, uint32_t g1, float* gk,
                                                  float* As, float* Cs, uint32_t* next, int lane)
{
    const int K = w.K, km = K - 2;
    const int ra = td.r[km], cols = td.d[km] * RB_;
    const uint32_t nK = (uint32_t)td.n[K - 1];
    for (;;) {   // groups are handed out through a shared counter: their row counts differ widely
        uint32_t j = 0;
        if (lane == 0) j = atomicAdd(next, 1u);
        j = __shfl_sync(0xffffffffu, j, 0);
        if (j >= g1) break;
        const uint32_t g = w.tnode[K - 1][j];   // units are cut from the digit-major order (see forward.cu)
        const uint32_t val = w.val[K - 1][g];
        const float* src = tt_left_operand(w, td, K - 1, g);
        for (int i = lane; i < M * ra; i += 32) {
            const int m = i / ra, a = i - m * ra;
            As[a * M + m] = __ldg(src + i);
        }
        __syncwarp();
        const uint32_t im = val % (uint32_t)td.n[km];
        tt_warp_mid_b<M, CPL, (MMA ? RB_ : 0)>(As, td.core[km] + (size_t)im * td.slice_floats[km], Cs, ra, cols, lane);
        __syncwarp();
        const uint32_t u0 = w.cstart[K - 1][g], u1 = w.cstart[K - 1][g + 1];
        if constexpr (MMA) {
            // two passes keep the register footprint low enough for twice the resident warps of one fused loop
            tt_warp_rows_dC_mma<PM, RB_>(w, td, u0, u1, val * nK, w.dP[K - 1] + (size_t)g * w.stride[K - 1], lane);
            tt_warp_rows_dG_mma<PM, RB_>(Cs, w, u0, u1, val * nK, gk, lane);
        } else {
            tt_warp_rows_dC<PM, RB_, TP>(w, td, u0, u1, val * nK, w.dP[K - 1] + (size_t)g * w.stride[K - 1], lane);
            tt_warp_rows_dG<PM, RB_, TP>(Cs, w, u0, u1, val * nK, gk, lane);
        }
        __syncwarp();
    }
}

// The fused-loop shapes with the intermediate products of NG = 16 / MROWS neighbouring groups formed together on the
// tensor cores, as in the forward sweep (quad_mid.cuh): one group at a time, every group read its whole slice of core
// K-1 (16 KB at rank 32) for a product of MROWS rows, which made the L1/L2 path the limit where groups hold few rows.
template <int PM, int RB_, int MROWS, int KTMAX, bool FEW>
__device__ __forceinline__ void tt_sweep_bwd_quad(const WsView& w, const TableDesc& td, uint32_t g1, float* gk, float* Cs4,
                                                  uint32_t* next, int lane)
{
    constexpr int COLS = PM / MROWS * RB_;   // d_{K-1} * r_{K-1}
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
        uint32_t gq = 0, valq = 0, imq = 0, u0q = 0, u1q = 0;
        const float* srcq = nullptr;
        if (lane < cnt) {
            gq = w.tnode[K - 1][base + lane];   // position in the digit-major order -> group
            valq = w.val[K - 1][gq];
            imq = valq % (uint32_t)td.n[km];
            srcq = tt_left_operand(w, td, K - 1, gq);
            u0q = w.cstart[K - 1][gq];
            u1q = w.cstart[K - 1][gq + 1];
        }
        tt_quad_mid<COLS, MROWS, KTMAX, RB_>(td.core[km], td.slice_floats[km], ra, cnt, imq, srcq, Cs4, lane);
        __syncwarp();
        for (int q = 0; q < cnt; ++q) {
            const uint32_t g = __shfl_sync(0xffffffffu, gq, q), val = __shfl_sync(0xffffffffu, valq, q);
            const uint32_t u0 = __shfl_sync(0xffffffffu, u0q, q), u1 = __shfl_sync(0xffffffffu, u1q, q);
            static_assert(PM == 8, "the fused loop takes C of 8 rows");
            tt_warp_rows_bwd_mma<RB_, RB_ + 4>(Cs4 + (size_t)q * (PM * (RB_ + 4)), w, td, u0, u1, val * nK,
                                                   w.dP[K - 1] + (size_t)g * w.stride[K - 1], gk, lane);
        }
        __syncwarp();
    }
}

// The same with the rows of the batch as one stream (stream.cuh).  Per step of four rows:
//   dC += sum_{row, j} dE[p][j] D[b][j]: k = (row, j), two k steps.  Lane t of a quad takes row t: k = t and t + 4 are j = 0, 1 in
//         the first step and 2, 3 in the second, so that a fragment is one 16-byte load.  C of 8 or 4 rows: transposed.
//   dG_K[i_K] += C^T . dE: n = (row, j), two tiles: n / 2 is the row (tt_stream_row), j = 2 (n % 2) + tile, so that an operand of both
//         tiles is one 8-byte load and a lane ends up with four neighbouring floats of one slice.
template <int PM, int RB_, int MROWS, int KTMAX, int PD, bool FEW>
__device__ __forceinline__ void tt_sweep_bwd_stream(const WsView& w, const TableDesc& td, uint32_t g1, float* gk, float* Cs4,
                                                    uint32_t* next, int lane)
{
    constexpr int COLS = PM / MROWS * RB_, NG = 16 / MROWS, CS = RB_ + 4;
    constexpr bool TR = PM < 16;                  // dC transposed: M = b, N = p
    constexpr bool KHALF = PM == 4;               // p = 4..7 of the one dG k step do not exist: zero operands
    constexpr int MT = TR ? 1 : PM / 16, NT = RB_ / 8;
    constexpr bool BHALF = RB_ == 8;              // b = 8..15 of the one row tile over b do not exist: zero operands, not stored
    constexpr int MT2 = BHALF ? 1 : RB_ / 16, KT2 = KHALF ? 1 : PM / 8;
    constexpr int DM = TR ? MT2 : MT, DN = TR ? 1 : NT;
    using Stream = RowStream<PM, RB_, NG, PD>;
    constexpr int EP = Stream::EP, DP = Stream::DP;
    const int K = w.K, km = K - 2, g = lane >> 2, t = lane & 3;
    const int ra = td.r[km];
    const uint32_t nK = (uint32_t)td.n[K - 1];
    const int rn = tt_stream_row(g >> 1), rc = tt_stream_row(t);   // dG: row of this lane's column n = g of dE; of its columns 2t, 2t + 1 of the result
    Stream rs(w.val[K], td.core[K - 1], Cs4 + NG * PM * CS, lane);
    uint32_t nbase = 0;
    if (lane == 0) nbase = atomicAdd(next, FEW ? next[1] : (uint32_t)NG);
    nbase = __shfl_sync(0xffffffffu, nbase, 0);
    uint32_t gq = (uint32_t)lane < (FEW ? next[1] : (uint32_t)NG) && nbase + lane < g1 ? w.tnode[K - 1][nbase + lane] : 0u;   // lane k: group k of the batch
    while (nbase < g1) {
        const int cnt = (int)min(FEW ? next[1] : (uint32_t)NG, g1 - nbase);
        uint32_t valq = 0, imq = 0, u0q = 0, u1q = 0;
        const float* srcq = nullptr;
        if (lane < cnt) {
            valq = w.val[K - 1][gq];
            imq = valq % (uint32_t)td.n[km];
            srcq = tt_left_operand(w, td, K - 1, gq);
            u0q = w.cstart[K - 1][gq];
            u1q = w.cstart[K - 1][gq + 1];
        }
        rs.begin(gq, u0q, u1q, valq * nK, lane);
        auto fill = [&]() { rs.fill(w.E, lane); };
        if constexpr (RB_ == 8) tt_quad_mid_fp32<RB_>(td.core[km], td.slice_floats[km], ra, cnt, imq, srcq, Cs4, lane, fill);
        else tt_quad_mid<COLS, MROWS, KTMAX, RB_>(td.core[km], td.slice_floats[km], ra, cnt, imq, srcq, Cs4, lane, fill);
        if (lane == 0) nbase = atomicAdd(next, FEW ? next[1] : (uint32_t)NG);
        nbase = __shfl_sync(0xffffffffu, nbase, 0);
        gq = (uint32_t)lane < (FEW ? next[1] : (uint32_t)NG) && nbase + lane < g1 ? w.tnode[K - 1][nbase + lane] : 0u;   // the next batch
        __syncwarp();
        Tf32Pair ct[MT2][KT2][4];   // A[m = b][k = p] = C[p][b] of the current group
        float dc[DM][DN][4];
        uint32_t cur = 0xffffffffu, chain = 0;
        bool folded = false;
        // dC of the group so far to dP (a chain of the tensor core's truncating additions ends here: the sum goes on in rounded fp32)
        auto hand_over = [&](uint32_t q) {
            float* dst = w.dP[K - 1] + (size_t)rs.groups()[32 + q] * w.stride[K - 1];
            if constexpr (TR) {
                if (2 * t < PM) {
#pragma unroll
                    for (int mt = 0; mt < DM; ++mt)
#pragma unroll
                        for (int x = 0; x < (BHALF ? 2 : 4); ++x) {
                            float* d = dst + (2 * t + (x & 1)) * RB_ + 16 * mt + g + 8 * (x >> 1);
                            *d = folded ? *d + dc[mt][0][x] : dc[mt][0][x];
                        }
                }
            } else {
#pragma unroll
                for (int mt = 0; mt < DM; ++mt)
#pragma unroll
                    for (int nt = 0; nt < DN; ++nt)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float2* d = reinterpret_cast<float2*>(dst + (16 * mt + 8 * h + g) * RB_ + 8 * nt + 2 * t);
                            float2 v = make_float2(dc[mt][nt][2 * h], dc[mt][nt][2 * h + 1]);
                            if (folded) { const float2 o = *d; v.x += o.x; v.y += o.y; }
                            *d = v;
                        }
            }
#pragma unroll
            for (int mt = 0; mt < DM; ++mt)
#pragma unroll
                for (int nt = 0; nt < DN; ++nt)
#pragma unroll
                    for (int x = 0; x < 4; ++x) dc[mt][nt][x] = 0.f;
            chain = 0;
        };
#pragma unroll
        for (int mt = 0; mt < DM; ++mt)
#pragma unroll
            for (int nt = 0; nt < DN; ++nt)
#pragma unroll
                for (int x = 0; x < 4; ++x) dc[mt][nt][x] = 0.f;
#pragma unroll 1
        for (int q = 0; q < cnt; ++q)   // groups without rows (dropped at the row capacity)
            if (rs.groups()[8 + q] == rs.groups()[16 + q]) hand_over(q);
        int slot = 0;
#pragma unroll 1
        for (uint32_t s = 0; s <= rs.steps; ++s) {
            const uint32_t qn = s < rs.steps ? *rs.group_rows(s) : 0xffu, q = qn & 255u, nr = qn >> 8;
            if (q != cur || chain >= 16) {
                if (cur != 0xffffffffu) hand_over(cur);
                if (s == rs.steps) break;
                folded = q == cur;
                if (q != cur) {
                    cur = q;
                    const float* Cs = Cs4 + q * (PM * CS);
#pragma unroll
                    for (int mt = 0; mt < MT2; ++mt)
#pragma unroll
                        for (int kt = 0; kt < KT2; ++kt) {
                            ct[mt][kt][0] = tt_split_tf32(Cs[(8 * kt + t) * CS + 16 * mt + g]);
                            ct[mt][kt][1] = tt_split_tf32(BHALF ? 0.f : Cs[(8 * kt + t) * CS + 16 * mt + g + 8]);
                            ct[mt][kt][2] = tt_split_tf32(KHALF ? 0.f : Cs[(8 * kt + t + 4) * CS + 16 * mt + g]);
                            ct[mt][kt][3] = tt_split_tf32(KHALF || BHALF ? 0.f : Cs[(8 * kt + t + 4) * CS + 16 * mt + g + 8]);
                        }
                }
            }
            const float* st = rs.wait(slot);
            if (nr <= 2) {
                // a step of one or two rows: half of the products, k = (row, j) and n = (row, j) in the order row, j.  (As four rows, two
                // of them zeros, a row's four terms went into dC as two sums, each truncated: gradients of the first core with one to
                // three rows per group 6 to 10 % further from 64 bits, 3.43e-7 instead of 3.13e-7 with C of 4 rows, rank 16.)
                float acc[MT2][4];
#pragma unroll
                for (int mt = 0; mt < MT2; ++mt)
#pragma unroll
                    for (int x = 0; x < 4; ++x) acc[mt][x] = 0.f;
                const float* El = st + (g >> 2) * EP + 4 * t + (g & 3);
#pragma unroll
                for (int kt = 0; kt < KT2; ++kt) {
                    const Tf32Pair b[2] = {tt_split_tf32(El[32 * kt]), tt_split_tf32(KHALF ? 0.f : El[32 * kt + 16])};
#pragma unroll
                    for (int mt = 0; mt < MT2; ++mt) tt_mma_3xtf32(acc[mt], ct[mt][kt], b);
                }
                const float* Et = st + 4 * g + t;
                const float* Dt = st + 4 * EP + 4 * g + t;
                if constexpr (TR) {
                    const bool on = PM == 8 || g < PM;
                    const Tf32Pair b[2] = {tt_split_tf32(on ? Et[0] : 0.f), tt_split_tf32(on ? Et[EP] : 0.f)};
#pragma unroll
                    for (int mt = 0; mt < MT2; ++mt) {
                        const Tf32Pair a[4] = {tt_split_tf32(Dt[64 * mt]), tt_split_tf32(BHALF ? 0.f : Dt[64 * mt + 32]),
                                               tt_split_tf32(Dt[DP + 64 * mt]), tt_split_tf32(BHALF ? 0.f : Dt[DP + 64 * mt + 32])};
                        tt_mma_3xtf32(dc[mt][0], a, b);
                    }
                } else {
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        const Tf32Pair a[4] = {tt_split_tf32(Et[64 * mt]), tt_split_tf32(Et[64 * mt + 32]),
                                               tt_split_tf32(Et[EP + 64 * mt]), tt_split_tf32(Et[EP + 64 * mt + 32])};
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            const Tf32Pair b[2] = {tt_split_tf32(Dt[32 * nt]), tt_split_tf32(Dt[DP + 32 * nt])};
                            tt_mma_3xtf32(dc[mt][nt], a, b);
                        }
                    }
                }
                if ((uint32_t)(t >> 1) < nr) {
                    float* dst = gk + (size_t)rs.ids(s)[t >> 1] * (RB_ * 4) + 4 * g + 2 * (t & 1);
#pragma unroll
                    for (int mt = 0; mt < MT2; ++mt) {
                        tt_red_v2(dst + 64 * mt, acc[mt][0], acc[mt][1]);
                        if (!BHALF) tt_red_v2(dst + 64 * mt + 32, acc[mt][2], acc[mt][3]);
                    }
                }
                chain += 1;
            } else {
                // ---- dG_K[i_K] += C^T . dE
                float acc[2][MT2][4];
    #pragma unroll
                for (int tile = 0; tile < 2; ++tile)
    #pragma unroll
                    for (int mt = 0; mt < MT2; ++mt)
    #pragma unroll
                        for (int x = 0; x < 4; ++x) acc[tile][mt][x] = 0.f;
                const float* El = st + rn * EP + 4 * t + 2 * (g & 1);
    #pragma unroll
                for (int kt = 0; kt < KT2; ++kt) {
                    const float2 e0 = *reinterpret_cast<const float2*>(El + 32 * kt);
                    const float2 e1 = KHALF ? make_float2(0.f, 0.f) : *reinterpret_cast<const float2*>(El + 32 * kt + 16);
                    const Tf32Pair b0[2] = {tt_split_tf32(e0.x), tt_split_tf32(e1.x)}, b1[2] = {tt_split_tf32(e0.y), tt_split_tf32(e1.y)};
    #pragma unroll
                    for (int mt = 0; mt < MT2; ++mt) {
                        tt_mma_3xtf32(acc[0][mt], ct[mt][kt], b0);
                        tt_mma_3xtf32(acc[1][mt], ct[mt][kt], b1);
                    }
                }
                // ---- dC += dE . D^T
                const float* Et = st + t * EP + 4 * g;
                const float* Dt = st + 4 * EP + t * DP + 4 * g;
                auto split4 = [](Tf32Pair (&d)[4], const float4& v) {
                    d[0] = tt_split_tf32(v.x); d[1] = tt_split_tf32(v.y); d[2] = tt_split_tf32(v.z); d[3] = tt_split_tf32(v.w);
                };
                if constexpr (TR) {
                    Tf32Pair e[4];   // dE[p = g] of row t, j = 0..3
                    split4(e, PM == 8 || g < PM ? *reinterpret_cast<const float4*>(Et) : make_float4(0.f, 0.f, 0.f, 0.f));
                    const Tf32Pair b0[2] = {e[0], e[1]}, b1[2] = {e[2], e[3]};
    #pragma unroll
                    for (int mt = 0; mt < MT2; ++mt) {
                        Tf32Pair x[4], y[4];
                        split4(x, *reinterpret_cast<const float4*>(Dt + 64 * mt));
                        split4(y, BHALF ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4*>(Dt + 64 * mt + 32));
                        const Tf32Pair a0[4] = {x[0], y[0], x[1], y[1]}, a1[4] = {x[2], y[2], x[3], y[3]};
                        tt_mma_3xtf32(dc[mt][0], a0, b0);
                        tt_mma_3xtf32(dc[mt][0], a1, b1);
                    }
                } else {
    #pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        Tf32Pair x[4], y[4];
                        split4(x, *reinterpret_cast<const float4*>(Et + 64 * mt));
                        split4(y, *reinterpret_cast<const float4*>(Et + 64 * mt + 32));
                        const Tf32Pair a0[4] = {x[0], y[0], x[1], y[1]}, a1[4] = {x[2], y[2], x[3], y[3]};
    #pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            Tf32Pair d[4];
                            split4(d, *reinterpret_cast<const float4*>(Dt + 32 * nt));
                            const Tf32Pair b0[2] = {d[0], d[1]}, b1[2] = {d[2], d[3]};
                            tt_mma_3xtf32(dc[mt][nt], a0, b0);
                            tt_mma_3xtf32(dc[mt][nt], a1, b1);
                        }
                    }
                }
                float* dst = gk + (size_t)rs.ids(s)[rc] * (RB_ * 4) + 4 * g;
    #pragma unroll
                for (int mt = 0; mt < MT2; ++mt)
    #pragma unroll
                    for (int h = 0; h < (BHALF ? 1 : 2); ++h)
                        tt_red_v4_if((uint32_t)rc < nr, dst + (16 * mt + 8 * h) * 4, acc[0][mt][2 * h], acc[1][mt][2 * h],
                                     acc[0][mt][2 * h + 1], acc[1][mt][2 * h + 1]);
                chain += 2;
            }
            __syncwarp();
            rs.stage(slot, w.E, lane);
            slot = slot + 1 == PD ? 0 : slot + 1;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
    }
}
#define BWD_RING 2   // steps in a warp's ring
template <int PM, int RB_, int MROWS>
struct BwdStream { static constexpr int FLOATS = 16 / MROWS * PM * (RB_ + 4) + RowStream<PM, RB_, 16 / MROWS, BWD_RING>::FLOATS; };   // per warp

// rank-64 four-core shape (wide.cuh).  dG_K: a warp takes one row, a lane two values of b over the 32 rows of C and dE.  dC (32 x
// 64) = sum over the group's rows of dE . D^T: two warps per group, half the columns each, as 3xTF32 tiles whose k is two rows
// by four columns, every pair of rows added in rounded fp32 (a group has up to n_K rows).
template <bool FEW>
__global__ void __launch_bounds__(WIDE_THREADS, 2) k_sweep_bwd_wide(WsView w, int vbase)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ WideBatch batches[2];
    float *Bs = sm, *As = Bs + 64 * WIDE_BP, *Cs = As + 8 * WIDE_GROUPS * WIDE_AP;
    const int t = w.vlist[vbase + (FEW ? blockIdx.x : blockIdx.y)], K = w.K, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const TableDesc& td = w.tdesc[t];
    uint32_t step;
    const uint2 rng = tt_sweep_unit<FEW>(w, t, WIDE_GROUPS, step);
    const int stripe = (blockIdx.x + blockIdx.y) % TT_STRIPES;
    float* gk = w.gpart + (size_t)stripe * w.gpart_stride + td.gpart_off;
    const uint32_t nK = (uint32_t)td.n[K - 1];
    WideLoop<true> loop(w, td, rng, batches, Bs, As, Cs);
    while (loop.next()) {
        const WideBatch& b = loop.batch();
        const uint32_t rows = wide_rows(b);
        float4* stage = reinterpret_cast<float4*>(As) + wid * 64;   // this warp's rows of dE, one at a time
        for (uint32_t r = wid; r < rows; r += WIDE_THREADS / 32) {
            uint32_t u;
            const int q = wide_row(b, r, u);
            __syncwarp();
            tt_cp_async16(stage + lane, reinterpret_cast<const float4*>(w.E + (size_t)u * w.D) + lane);
            const uint32_t iK = w.val[K][u] - b.val[q] * nK;
            asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            const float* c = Cs + q * (32 * WIDE_CP) + lane;
            float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
#pragma unroll 8
            for (int p = 0; p < 32; ++p) {
                const float4 d = stage[p];
                const float y0 = c[p * WIDE_CP], y1 = c[p * WIDE_CP + 32];
                x0.x = fmaf(y0, d.x, x0.x); x0.y = fmaf(y0, d.y, x0.y); x0.z = fmaf(y0, d.z, x0.z); x0.w = fmaf(y0, d.w, x0.w);
                x1.x = fmaf(y1, d.x, x1.x); x1.y = fmaf(y1, d.y, x1.y); x1.z = fmaf(y1, d.z, x1.z); x1.w = fmaf(y1, d.w, x1.w);
            }
            float* dst = gk + (size_t)iK * 256 + lane * 4;
            tt_red_v4(dst, x0.x, x0.y, x0.z, x0.w);
            tt_red_v4(dst + 128, x1.x, x1.y, x1.z, x1.w);
        }
        const int q = wid >> 1, n0 = 32 * (wid & 1), g = lane >> 2, j = lane & 3;
        if (b.im[q] != 0xffffffffu) {
            float sum[2][4][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int x = 0; x < 4; ++x) sum[mt][nt][x] = 0.f;
            const uint32_t u1 = b.u1[q], row_base = b.val[q] * nK;
#pragma unroll 1
            for (uint32_t u = b.u0[q]; u < u1; u += 2) {
                const bool two = u + 1 < u1;
                const float* dE = w.E + (size_t)u * w.D + 4 * g + j;
                const float* D0 = td.core[K - 1] + (size_t)(w.val[K][u] - row_base) * 256 + 4 * (n0 + g) + j;
                const float* D1 = td.core[K - 1] + (size_t)(w.val[K][two ? u + 1 : u] - row_base) * 256 + 4 * (n0 + g) + j;
                float e[2][4], d[4][2];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    e[mt][0] = __ldg(dE + 64 * mt);
                    e[mt][1] = __ldg(dE + 64 * mt + 32);
                    e[mt][2] = two ? __ldg(dE + w.D + 64 * mt) : 0.f;
                    e[mt][3] = two ? __ldg(dE + w.D + 64 * mt + 32) : 0.f;
                }
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) { d[nt][0] = __ldg(D0 + 32 * nt); d[nt][1] = __ldg(D1 + 32 * nt); }
                Tf32Pair a[2][4];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int x = 0; x < 4; ++x) a[mt][x] = tt_split_tf32(e[mt][x]);
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    Tf32Pair f[2] = {tt_split_tf32(d[nt][0]), tt_split_tf32(d[nt][1])};
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) tt_mma_3xtf32_rounded(sum[mt][nt], a[mt], f);
                }
            }
            float* dst = w.dP[K - 1] + (size_t)b.g[q] * w.stride[K - 1] + n0 + 2 * j;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    *reinterpret_cast<float2*>(dst + (16 * mt + g) * 64 + 8 * nt) = make_float2(sum[mt][nt][0], sum[mt][nt][1]);
                    *reinterpret_cast<float2*>(dst + (16 * mt + g + 8) * 64 + 8 * nt) = make_float2(sum[mt][nt][2], sum[mt][nt][3]);
                }
        }
    }
}

// One CTA (4 warps) per work unit (table, q); last-core gradients go to one of TT_STRIPES L2-resident partial
// copies with vector reductions, added up in fixed stripe order by k_reduce_gpart.
template <int V, bool FEW>
__global__ void __launch_bounds__(128, V == 5 ? 6 : V == 1 || V == 8 ? 4 : V == 2 || V == 6 || V == 9 ? 5 : 0) k_sweep_bwd(WsView w, int pl_floats, int c_floats, int vbase)
{
    tt_pdl_enter();
    extern __shared__ __align__(16) float sm[];
    const int t = w.vlist[vbase + (FEW ? blockIdx.x : blockIdx.y)];
    const TableDesc& td = w.tdesc[t];
    const int stripe = (blockIdx.x + blockIdx.y) % TT_STRIPES;
    float* gk = w.gpart + (size_t)stripe * w.gpart_stride + td.gpart_off;
    __shared__ uint32_t next[2];   // the CTA's next group, groups that a warp takes at a time
    uint32_t step;
    const uint2 rng = tt_sweep_unit<FEW>(w, t, V < 5 ? 4 : 8, step);
    const uint32_t g1 = rng.y;
    if (threadIdx.x == 0) { next[0] = rng.x; next[1] = step; }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float* As = sm + (size_t)wid * (pl_floats + c_floats);
    float* Cs = As + pl_floats;
    if (V == 0) tt_sweep_bwd_fast<16, 32, 4, 4, 1, true>(w, td, g1, gk, As, Cs, next, lane);
    if (V == 1) tt_sweep_bwd_stream<16, 16, 4, 4, BWD_RING, FEW>(w, td, g1, gk, sm + wid * BwdStream<16, 16, 4>::FLOATS, next, lane);
    if (V == 2) tt_sweep_bwd_stream<16, 8, 4, 4, BWD_RING, FEW>(w, td, g1, gk, sm + wid * BwdStream<16, 8, 4>::FLOATS, next, lane);
    if (V == 3) tt_sweep_bwd_fast<32, 32, 4, 4, 2, true>(w, td, g1, gk, As, Cs, next, lane);
    if (V == 5) tt_sweep_bwd_quad<8, 32, 2, 4, FEW>(w, td, g1, gk, sm + (size_t)wid * (8 * 8 * 36), next, lane);
    if (V == 6) tt_sweep_bwd_stream<8, 16, 2, 4, BWD_RING, FEW>(w, td, g1, gk, sm + wid * BwdStream<8, 16, 2>::FLOATS, next, lane);
    if (V == 7) tt_sweep_bwd_fast<8, 8, 2, 2, 1, false>(w, td, g1, gk, As, Cs, next, lane);   // 8 x 8: the FP32 pipe wins (51 us against 57 with streamed rows; 8 tables, 5 M lookups 172 / 184)
    if (V == 8) tt_sweep_bwd_stream<4, 32, 2, 4, BWD_RING, FEW>(w, td, g1, gk, sm + wid * BwdStream<4, 32, 2>::FLOATS, next, lane);
    if (V == 9) tt_sweep_bwd_stream<4, 16, 2, 4, BWD_RING, FEW>(w, td, g1, gk, sm + wid * BwdStream<4, 16, 2>::FLOATS, next, lane);
    if (V == 10) tt_sweep_bwd_fast<4, 8, 2, 2, 1, false>(w, td, g1, gk, As, Cs, next, lane);
}

// fixed-order sum of the partial copies of the last core's gradient
__global__ void __launch_bounds__(256) k_reduce_gpart(WsView w)
{
    tt_pdl_enter();
    const int t = blockIdx.y;
    const TableDesc& td = w.tdesc[t];
    const int kl = w.K - 1;
    const int64_t n = td.core_floats[kl];
    const float* src = w.gpart + td.gpart_off;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < TT_STRIPES; ++q) s += src[(size_t)q * w.gpart_stride + i];
        td.grad[kl][i] = s;
        if (w.fused_lr != 0.f) td.core[kl][i] = td.core[kl][i] - w.fused_lr * s;   // nothing reads the last core after the sweeps
    }
}

template <int V>
static cudaError_t launch_sweep_bwd(tt_emb* h, int max_pl, int max_c, cudaStream_t s)
{
    const int n = h->vcount[V + 1];
    if (n == 0) return cudaSuccess;
    [[maybe_unused]] const bool few = tt_few_groups(h);
    // tensor-core variants keep C with padded rows (stride r_{K-1} + 8 floats)
    if (V == 0) max_c = 16 * (32 + 8);
    if (V == 3) max_c = 32 * (32 + 8);
    size_t smem = (size_t)4 * (max_pl + max_c) * sizeof(float);
    if (V == 5) smem = (size_t)4 * 8 * 8 * 36 * sizeof(float);    // eight C tiles per warp, rows padded by four floats
    if (V == 6) smem = (size_t)4 * BwdStream<8, 16, 2>::FLOATS * sizeof(float);
    if (V == 8) smem = (size_t)4 * BwdStream<4, 32, 2>::FLOATS * sizeof(float);
    if (V == 9) smem = (size_t)4 * BwdStream<4, 16, 2>::FLOATS * sizeof(float);
    if (V == 1) smem = (size_t)4 * BwdStream<16, 16, 4>::FLOATS * sizeof(float);
    if (V == 2) smem = (size_t)4 * BwdStream<16, 8, 4>::FLOATS * sizeof(float);
    cudaError_t e;
    if ((e = tt_stage_begin(h, 9 + TT_NUM_VARIANTS + 1 + V + 1, s)) != cudaSuccess) return e;
    if constexpr (V < 0) {
        int c_floats;
        if (const int dk = gen_odd_factor(h, c_floats)) {
            auto kern = dk == 1 ? k_sweep_bwd_odd<1> : dk == 2 ? k_sweep_bwd_odd<2> : dk == 3 ? k_sweep_bwd_odd<3>
                      : dk == 5 ? k_sweep_bwd_odd<5> : dk == 6 ? k_sweep_bwd_odd<6> : k_sweep_bwd_odd<7>;
            smem = (size_t)(2 * c_floats + gen_stage_rows(h->D) * gen_stage_pitch(h->D)) * sizeof(float);
            if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
            if ((e = tt_launch_pdl(kern, dim3(h->units_per_table, n), dim3(GEN_ODD_THREADS), smem, s, h->v, h->vbase[0], c_floats)) != cudaSuccess) return e;
            tt_note_launch();
            if ((e = tt_stage_end(h, 9 + TT_NUM_VARIANTS + 1 + V + 1, s)) != cudaSuccess) return e;
            return cudaGetLastError();
        }
        smem = 2 * GEN_C_FLOATS * sizeof(float);
        if ((e = cudaFuncSetAttribute(k_sweep_bwd_any, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(k_sweep_bwd_any, dim3(h->units_per_table, n), dim3(GEN_THREADS), smem, s, h->v, h->vbase[0])) != cudaSuccess) return e;
    } else if constexpr (V == 4) {
        auto kern = few ? k_sweep_bwd_wide<true> : k_sweep_bwd_wide<false>;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WIDE_SMEM)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(kern, few ? dim3(n, h->sweep_ctas) : dim3(h->units_per_table, n), dim3(WIDE_THREADS), WIDE_SMEM, s, h->v, h->vbase[V + 1])) != cudaSuccess) return e;
    } else {
        auto kern = few ? k_sweep_bwd<V, true> : k_sweep_bwd<V, false>;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(kern, few ? dim3(n, h->sweep_ctas) : dim3(h->units_per_table, n), dim3(128), smem, s, h->v, max_pl, max_c, h->vbase[V + 1])) != cudaSuccess) return e;
    }
    tt_note_launch();
    if ((e = tt_stage_end(h, 9 + TT_NUM_VARIANTS + 1 + V + 1, s)) != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t tt_launch_bwd_contraction(tt_emb* h, cudaStream_t s)
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
    // four cores: the digit-major list of level 2 is made beside the sweeps, as far as the scan's space is free (the segment starts are done
    // with); the middle level waits for it.  Five short kernels on the way of the call otherwise: 65 k lookups, rank 64, call 380 to 367 us.
    // With several shape variants the first one's sweep follows the list on its stream.  The sweeps on the other streams only, backward, us,
    // behind it / not: one table of rank 64 and one of any shape, 33 k lookups 230 / 246, a third of any shape 269 / 283; two of rank 64 and
    // one of any shape, 12 k 176 / 166.
    if (h->K == 4 && !h->serial) {
        if ((e = tt_fork(h, s, 1)) != cudaSuccess) return e;
        if ((e = tt_launch_tlist(h, 2, h->side[0])) != cudaSuccess) return e;
    }
    // P_k of the levels below K-1 are still in pbuf from the forward (K = 4 only)
    // tables of different shape variants are independent: their kernels run side by side on forked streams
    int nvar = 0;
    for (int vi = 0; vi <= TT_NUM_VARIANTS; ++vi) nvar += h->vcount[vi] > 0 ? 1 : 0;
    const bool fork = nvar > 1 && !h->serial;
    if (fork && (e = tt_fork(h, s, 4)) != cudaSuccess) return e;
    int slot = 0;
    auto next_stream = [&](int vi) { return (fork && h->vcount[vi] > 0) ? h->side[(slot++) & 3] : s; };
    if ((e = launch_sweep_bwd<-1>(h, max_pl, max_c, next_stream(0))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<0>(h, max_pl, max_c, next_stream(1))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<1>(h, max_pl, max_c, next_stream(2))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<2>(h, max_pl, max_c, next_stream(3))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<3>(h, max_pl, max_c, next_stream(4))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<4>(h, max_pl, max_c, next_stream(5))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<5>(h, max_pl, max_c, next_stream(6))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<6>(h, max_pl, max_c, next_stream(7))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<7>(h, max_pl, max_c, next_stream(8))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<8>(h, max_pl, max_c, next_stream(9))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<9>(h, max_pl, max_c, next_stream(10))) != cudaSuccess) return e;
    if ((e = launch_sweep_bwd<10>(h, max_pl, max_c, next_stream(11))) != cudaSuccess) return e;
    if (fork && (e = tt_join(h, s, 4)) != cudaSuccess) return e;
    if ((e = tt_launch_pdl(k_reduce_gpart, dim3(32, h->T), dim3(256), 0, s, w)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- 4. middle cores

// ---- tensor-core middle-core backward (P_{k-1} = 4 or 2 rows, r_{k-1} in {16,32}, d_k * r_k in {32,64,128}) ----
//
// One CTA of 4 warps per (table, slice i_k).  The nodes with digit i_k arrive in ascending parent order from the
// digit-major list, 16 or 32 stacked rows (node, m) per pass: NQ = 4..16 nodes, staged with cp.async into padded
// shared-memory tiles (two stages, two barriers per pass), and both products run as 3xTF32 m16n8k8 tiles (mma.cuh):
//   dG_k[a][c] += sum_{node, m} P_{k-1}[node][m][a] * dP_k[node][m][c]   M = a, N = c, K = 8 stacked rows (node, m);
//                 a warp owns COLS/4 columns c of the slice, accumulators stay in registers over the whole list
//   Y[node][m][a] = sum_c dP_k[node][m][c] * G_k[a][c]                   M = 16 stacked rows, N = 8 values of a,
//                 K = c; the slice sits unsplit in shared memory (its 64 registers of split fragments per thread
//                 held the kernel at three CTAs per SM; at ~95 registers five are resident);
//                 warp -> (n-tile of a, tile of sixteen stacked rows)
// k_mid_sum then adds the Y rows of each parent's (contiguous) children.
// Row strides RA + 8 and COLS + 8 floats make every fragment load from shared memory conflict-free or 2-way.
// The tensor core adds into its fp32 accumulator with truncation, so an accumulation chain of N products drifts by
// up to N * 2^-24 of the sum; the dG accumulators are therefore folded into running sums (a rounded fp32
// add into the CTA's own gradient slice, which stays in L2) every eighth pass, which keeps every chain at 48 or 96
// products whatever the length of the node list.
template <int M, int RA, int COLS, int NQF = 1>
constexpr size_t tt_mid_smem_bytes()
{
    constexpr int NQ = NQF * 512 / (RA * M);
    return sizeof(float) * (size_t)(2 * NQ * M * (RA + 8) + 2 * NQ * M * (COLS + 8) + RA * (COLS + 4));
}

template <int M, int RA, int COLS, int NQF = 1>   // M = P_{k-1}: 4 or 2 rows per node; NQF: 2 = twice the nodes per pass
__global__ void __launch_bounds__(128, 5) k_mid_mma(WsView w, int k, int variant, int lbase)
{
    tt_pdl_enter();
    static_assert((M == 4 || M == 2) && (RA == 8 || RA % 16 == 0) && (COLS % 32 == 0 || COLS == 16), "rows per node; r_{k-1}; columns per warp");
    static_assert(NQF == 1 || NQF == 2, "one or two Y row tiles per warp");
    constexpr int NQ = NQF * 512 / (RA * M), AP = RA + 8, CP = COLS + 8;   // NQ * M = 16, 32 or 64 stacked rows per pass (x NQF)
    constexpr bool AHALF = RA == 8;          // dG: a = 8..15 of the one m-tile do not exist: zero operands, not stored
    constexpr int MT = AHALF ? 1 : RA / 16;  // dG: m-tiles over a
    constexpr int CW = COLS >= 32 ? COLS / 4 : 8;   // dG: columns per warp (16 columns: warps 0 and 1 only)
    constexpr int NTW = CW / 8;              // dG: n-tiles per warp
    constexpr int NTY = RA / 8;              // Y: n-tiles over a (4 or 2); NQ * M / 16 row tiles; NTY * NQ * M / 16 = 4 NQF tasks, NQF per warp
    constexpr int KTY = COLS / 8;            // Y: k steps over c
    extern __shared__ __align__(16) float mid_sm[];   // [2][NQ M AP] P rows, [2][NQ M CP] dP rows, [RA][COLS + 4] slice (tt_mid_smem_bytes)
    float* const sA = mid_sm;
    float* const sD = sA + 2 * NQ * M * AP;
    const int t_ = w.vlist[lbase + blockIdx.y];   // the tables of this variant, largest first: their long node lists start early
    const TableDesc& td = w.tdesc[t_];
    const int kc = k - 1;
    if (td.midfast[k] != variant || (int)blockIdx.x >= td.n[kc]) return;
    const uint32_t ik = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
    const float* __restrict__ Bsl = td.core[kc] + (size_t)ik * td.slice_floats[kc];
    // Y: this warp's n-tile of a and its four nodes
    const int ynt = wid % NTY, yrt0 = wid / NTY;   // task wid + 4 yi: the same n-tile, row tile yrt0 + yi * 4 / NTY
    // the slice G_k[i_k] for the Y product: unsplit in shared memory (row pitch COLS + 4: the fragment loads of a warp hit
    // 32 different banks), split at every use: registers for a fifth CTA per SM count for more than the 2 x 3 integer
    // operations per fragment
    constexpr int BP = COLS + 4;
    float* const sB = sD + 2 * NQ * M * CP;
    for (int i = tid; i < RA * (COLS / 4); i += 128) {
        const int a_ = i / (COLS / 4), c4 = i - a_ * (COLS / 4);
        tt_cp_async16(&sB[a_ * BP + 4 * c4], reinterpret_cast<const float4*>(Bsl + (size_t)a_ * COLS) + c4);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    // (asynchronous, so that the look-ups below do not queue behind it; it is the oldest copy group, so the wait for the
    // first pass's rows covers it, and the barrier after that wait orders it before its first use)
    const float* const sBw = sB + (8 * ynt + g) * BP + t;
    float acc[MT][NTW][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NTW; ++nt) { acc[mt][nt][0] = 0.f; acc[mt][nt][1] = 0.f; acc[mt][nt][2] = 0.f; acc[mt][nt][3] = 0.f; }
    // fold: this CTA is the only writer of its slice of the gradient, so the running sums live there (L2) instead of
    // in a second register set; each thread adds its accumulators to the elements it owns
    float* const gdst = td.grad[kc] + (size_t)ik * td.slice_floats[kc];
    bool first_fold = true;
    // last: the sums are final; the fused update of this CTA's slice goes with them (its fragments were read at the start,
    // and no other CTA or later kernel of the backward reads this slice)
    float* const cdst = td.core[kc] + (size_t)ik * td.slice_floats[kc];
    auto fold = [&](bool last) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            // all loads of a row tile first, then the sums and stores: one round trip per tile instead of one per
            // column block (the compiler cannot move a load above a store it cannot tell apart)
            float2 v0[NTW], v1[NTW], u0[NTW], u1[NTW];
            const bool upd = last && w.fused_lr != 0.f;
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt) {
                const int c = wid * CW + 8 * nt + 2 * t;
                v0[nt] = make_float2(0.f, 0.f); v1[nt] = v0[nt]; u0[nt] = v0[nt]; u1[nt] = v0[nt];
                if (c >= COLS) continue;     // this warp owns no columns of the slice gradient
                const size_t o0 = (size_t)(16 * mt + g) * COLS + c, o1 = (size_t)(16 * mt + g + 8) * COLS + c;
                if (!first_fold) {
                    v0[nt] = *reinterpret_cast<const float2*>(gdst + o0);
                    if (!AHALF) v1[nt] = *reinterpret_cast<const float2*>(gdst + o1);
                }
                if (upd) {   // the slice as it was read at the start (nobody else writes it): from its shared-memory copy
                    u0[nt] = *reinterpret_cast<const float2*>(sB + (16 * mt + g) * BP + c);
                    if (!AHALF) u1[nt] = *reinterpret_cast<const float2*>(sB + (16 * mt + g + 8) * BP + c);
                }
            }
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt) {
                const int c = wid * CW + 8 * nt + 2 * t;
                if (c >= COLS) continue;
                const size_t o0 = (size_t)(16 * mt + g) * COLS + c, o1 = (size_t)(16 * mt + g + 8) * COLS + c;
                v0[nt].x += acc[mt][nt][0]; v0[nt].y += acc[mt][nt][1]; v1[nt].x += acc[mt][nt][2]; v1[nt].y += acc[mt][nt][3];
                *reinterpret_cast<float2*>(gdst + o0) = v0[nt];
                if (!AHALF) *reinterpret_cast<float2*>(gdst + o1) = v1[nt];
                if (upd) {
                    u0[nt].x = u0[nt].x - w.fused_lr * v0[nt].x; u0[nt].y = u0[nt].y - w.fused_lr * v0[nt].y;
                    *reinterpret_cast<float2*>(cdst + o0) = u0[nt];
                    if (!AHALF) {
                        u1[nt].x = u1[nt].x - w.fused_lr * v1[nt].x; u1[nt].y = u1[nt].y - w.fused_lr * v1[nt].y;
                        *reinterpret_cast<float2*>(cdst + o1) = u1[nt];
                    }
                }
                acc[mt][nt][0] = 0.f; acc[mt][nt][1] = 0.f; acc[mt][nt][2] = 0.f; acc[mt][nt][3] = 0.f;
            }
        }
        first_fold = false;
    };
    const uint32_t space = td.prefix_space[k - 1];
    const uint32_t j0 = tt_trank(w, td, k, ik * space), j1 = tt_trank(w, td, k, (ik + 1) * space);
    const int strideY = w.stride[k - 1];
    const uint32_t passes = (j1 - j0 + NQ - 1) / NQ;
    // The node ids of a pass and the addresses of the nodes' left operands are looked up two passes ahead by NQ threads
    // (digit-major list -> node -> prefix value or parent -> operand: a chain of dependent loads) and handed to the
    // CTA through a ring in shared memory, so that staging a pass starts with its cp.async instructions.
    __shared__ uint32_t s_node[3][NQ];
    __shared__ const float* s_left[3][NQ];
    uint32_t pre_node = 0xffffffffu;
    const float* pre_left = nullptr;
    auto lookup_ids = [&](uint32_t r) {          // into registers (threads 0..NQ-1)
        pre_node = 0xffffffffu;
        pre_left = nullptr;
        if (tid < NQ && j0 + r * NQ + tid < j1) {
            pre_node = w.tnode[k][j0 + r * NQ + tid];
            pre_left = tt_left_operand(w, td, k, pre_node);
        }
    };
    auto publish_ids = [&](uint32_t r) {         // registers -> ring slot of pass r
        if (tid < NQ) { s_node[r % 3u][tid] = pre_node; s_left[r % 3u][tid] = pre_left; }
    };
    // stage the NQ nodes of pass r (missing nodes of the last pass are zero-filled)
    auto issue = [&](uint32_t r) {
        const int st = (int)(r & 1u);
        const uint32_t* ids = s_node[r % 3u];
        const float* const* lefts = s_left[r % 3u];
        for (int i = tid; i < NQ * M * (COLS / 4); i += 128) {   // dP_k rows: M * COLS / 4 float4 per node
            const int q = i / (M * (COLS / 4)), rem = i - q * (M * (COLS / 4)), m = rem / (COLS / 4), c4 = rem - m * (COLS / 4);
            float4* dst = reinterpret_cast<float4*>(&sD[st * NQ * M * CP + (q * M + m) * CP + 4 * c4]);
            const uint32_t v = ids[q];
            if (v != 0xffffffffu) tt_cp_async16(dst, reinterpret_cast<const float4*>(w.dP[k] + (size_t)v * w.stride[k] + m * COLS) + c4);
            else *dst = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int i = tid; i < NQ * M * (RA / 4); i += 128) {     // P_{k-1} of the parent: M * RA / 4 float4 per node
            const int q = i / (M * (RA / 4)), rem = i - q * (M * (RA / 4)), m = rem / (RA / 4), a4 = rem - m * (RA / 4);
            float4* dst = reinterpret_cast<float4*>(&sA[st * NQ * M * AP + (q * M + m) * AP + 4 * a4]);
            if (ids[q] != 0xffffffffu) tt_cp_async16(dst, reinterpret_cast<const float4*>(lefts[q] + m * RA) + a4);
            else *dst = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // passes 0 and 1 are looked up side by side (threads 0..NQ-1 and NQ..2NQ-1): one chain of round trips, not two
    if (tid < 2 * NQ) {
        const uint32_t r = (uint32_t)tid / NQ, q = (uint32_t)tid % NQ;
        uint32_t nd = 0xffffffffu;
        const float* lf = nullptr;
        if (j0 + r * NQ + q < j1) {
            nd = w.tnode[k][j0 + r * NQ + q];
            lf = tt_left_operand(w, td, k, nd);
        }
        s_node[r][q] = nd;
        s_left[r][q] = lf;
    }
    __syncthreads();
    if (passes > 0) issue(0);
    for (uint32_t r = 0; r < passes; ++r) {
        lookup_ids(r + 2);          // in flight while this pass is staged and computed; published at the end of the iteration
        if (r + 1 < passes) {
            issue(r + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float* A_ = sA + (r & 1u) * (NQ * M * AP);
        const float* D_ = sD + (r & 1u) * (NQ * M * CP);
        // ---- dG: eight stacked rows (node, m) give k = 8
#pragma unroll
        for (int p = 0; p < NQ * M / 8; ++p) {
            const float* Aa = A_ + (8 * p + t) * AP;       // stacked row 8p + t:     node (8p + t) / M, row (8p + t) % M
            const float* Ab = A_ + (8 * p + t + 4) * AP;   // stacked row 8p + t + 4
            if (wid * CW >= COLS) break;     // this warp owns no columns of the slice gradient
            const float* Da = D_ + (8 * p + t) * CP + wid * CW + g;
            const float* Db = D_ + (8 * p + t + 4) * CP + wid * CW + g;
            Tf32Pair a[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                a[mt][0] = tt_split_tf32(Aa[16 * mt + g]);
                a[mt][1] = tt_split_tf32(AHALF ? 0.f : Aa[16 * mt + g + 8]);
                a[mt][2] = tt_split_tf32(Ab[16 * mt + g]);
                a[mt][3] = tt_split_tf32(AHALF ? 0.f : Ab[16 * mt + g + 8]);
            }
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt) {
                Tf32Pair b[2];
                b[0] = tt_split_tf32(Da[8 * nt]);
                b[1] = tt_split_tf32(Db[8 * nt]);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) tt_mma_3xtf32(acc[mt][nt], a[mt], b);
            }
        }
        // ---- Y of this warp's sixteen stacked rows (NQF times) and eight values of a
#pragma unroll
        for (int yi = 0; yi < NQF; ++yi) {
            const int yrt = yrt0 + yi * (4 / NTY);
            float y[4] = {0.f, 0.f, 0.f, 0.f};
            const float* Ra = D_ + (16 * yrt + g) * CP;       // row g of the tile: stacked row 16 yrt + g
            const float* Rb = D_ + (16 * yrt + g + 8) * CP;   // row g + 8
#pragma unroll
            for (int kt = 0; kt < KTY; ++kt) {
                Tf32Pair a[4];
                a[0] = tt_split_tf32(Ra[8 * kt + t]);
                a[1] = tt_split_tf32(Rb[8 * kt + t]);
                a[2] = tt_split_tf32(Ra[8 * kt + t + 4]);
                a[3] = tt_split_tf32(Rb[8 * kt + t + 4]);
                Tf32Pair by[2];
                by[0] = tt_split_tf32(sBw[8 * kt]);
                by[1] = tt_split_tf32(sBw[8 * kt + 4]);
                tt_mma_3xtf32(y, a, by);
            }
            const uint32_t ja = j0 + r * NQ + (16 * yrt + g) / M, jb2 = j0 + r * NQ + (16 * yrt + g + 8) / M;
            const int ma = (16 * yrt + g) % M;   // the same row of P for g and g + 8 (M divides 8)
            if (ja < j1) {
                const uint32_t v = s_node[r % 3u][(16 * yrt + g) / M];
                *reinterpret_cast<float2*>(&w.Y[k][(size_t)v * strideY + ma * RA + 8 * ynt + 2 * t]) = make_float2(y[0], y[1]);
            }
            if (jb2 < j1) {
                const uint32_t v = s_node[r % 3u][(16 * yrt + g + 8) / M];
                *reinterpret_cast<float2*>(&w.Y[k][(size_t)v * strideY + ma * RA + 8 * ynt + 2 * t]) = make_float2(y[2], y[3]);
            }
        }
        if ((r & (8u / NQF - 1u)) == 8u / NQF - 1u) fold(false);   // rounded running sums every eighth pass (fourth with twice the nodes)
        publish_ids(r + 2);   // its ring slot held pass r - 1
        __syncthreads();   // everyone is done with this stage before pass r + 2 overwrites it
    }
    if (passes == 0) {   // no pass has waited for the slice copy
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    }
    fold(true);   // also writes the zeros of a slice without nodes
}

// ---- tensor-core middle-core backward for every other shape (any M = P_{k-1}, r_{k-1}, d_k * r_k) ----
//
// The same two products as k_mid_mma, cut into 64 x 64 output tiles so that wide slices spread over the SMs (rank 64:
// 64 slices of 64 x 256, i.e. 256 tiles of dG) and narrow ones fit one tile:
//   z < dgz   one tile of dG_k[i_k]: 64 values of a by 64 columns; k runs over the slice's stacked rows (node, m), 32 per
//             pass, staged with cp.async in two buffers, row addresses looked up two passes ahead
//   z >= dgz  Y: tiles of 64 stacked rows by 64 values of a, dealt out to the slice's `yctas` CTAs; k runs over the
//             columns, 32 per pass.  FOLD: to the CTAs of dG, after their tile
// A warp owns a 32 x 32 quarter of the tile (tiles.cuh; 16 fragment loads per k step for 8 tile products of 3xTF32); row
// tiles and column blocks outside the shape are skipped.  No fused update of the slice: the Y CTAs of other tiles still read it.
// Bound by the operand path (16 fragment loads for 24 tensor instructions) and, for short node lists, by a CTA's look-ups.
// Middle stage, 2x4x4x4 with rank 64 (65 536 lookups): 5.05 ms with one FP32 thread per output element over the whole
// node list, 0.16 ms as tiles; 3x3x5 with ranks 6 and 4 (4 tables, 1 M lookups): 0.41 and 0.06 ms.
template <bool FOLD, bool WHOLE>
__global__ void __launch_bounds__(128, 4) k_mid_tile(WsView w, int k, int lbase, int dgz, int yctas)
{
    tt_pdl_enter();
    __shared__ __align__(16) float sm[2 * 2 * MT_EDGE * MT_PC];   // = 2 * 2 * MT_KROWS * MT_PA
    static_assert(MT_EDGE * MT_PC == MT_KROWS * MT_PA, "both roles stage the same number of floats");
    constexpr int STAGE = MT_EDGE * MT_PC;
    const TableDesc& td = w.tdesc[w.vlist[lbase + blockIdx.y]];
    const int kc = k - 1;
    if ((int)blockIdx.x >= td.n[kc]) return;
    const uint32_t ik = blockIdx.x;
    const int M = td.P[kc], ra = td.r[kc], cols = td.d[kc] * td.r[kc + 1];
    const bool vec = (ra & 3) == 0 && (cols & 3) == 0;   // then every row, node and slice starts on a 16-byte boundary
    const uint32_t space = td.prefix_space[k - 1];
    const uint32_t j0 = tt_trank(w, td, k, ik * space), j1 = tt_trank(w, td, k, (ik + 1) * space);
    const uint64_t R = tt_stacked_rows(j1 - j0, M);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
    const int wr = wid >> 1, wc = wid & 1;               // this warp's quarter
    const int ach = (ra + MT_EDGE - 1) / MT_EDGE;
    float sum[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[mt][nt][i] = 0.f;

    const int cch = (cols + MT_EDGE - 1) / MT_EDGE;
    if ((int)blockIdx.z < (FOLD ? min(dgz, ach * cch) : dgz)) {
        // ------------------------------------------------------------------------------ a tile of the slice gradient
        if (!FOLD && (int)blockIdx.z >= ach * cch) return;
        const int a0 = (int)blockIdx.z / cch * MT_EDGE, c0 = (int)blockIdx.z % cch * MT_EDGE;
        const int mtl = min(2, max(0, (ra - a0 - 32 * wr + 15) / 16)), ntl = min(4, max(0, (cols - c0 - 32 * wc + 7) / 8));
        __shared__ const float* s_a[3][MT_KROWS];
        __shared__ const float* s_d[3][MT_KROWS];
        const uint64_t passes = (R + MT_KROWS - 1) / MT_KROWS;
        // this lane's row of a pass of 32 rows (a warp looks up one pass); the first of the passes that the warp looks up
        StackedRow at = tt_stacked_row((uint64_t)(wid < 2 ? wid : 0) * MT_KROWS + lane, M);
        auto lookup = [&](const float*& pa, const float*& pd) {
            pa = nullptr; pd = nullptr;
            if (at.node < j1 - j0) {
                const uint32_t v = w.tnode[k][j0 + at.node];
                pa = tt_left_operand(w, td, k, v) + (size_t)at.m * ra + a0;
                pd = w.dP[k] + (size_t)v * w.stride[k] + (size_t)at.m * cols + c0;
            }
        };
        // the pass's buffer, and its addresses in the ring of three
        auto issue = [&](int buf, int ring) {
            float* st = sm + buf * (2 * STAGE);
            tt_stage_rows<MT_KROWS, MT_EDGE / 4>(st, MT_PA, s_a[ring], 0, ra - a0, vec);
            tt_stage_rows<MT_KROWS, MT_EDGE / 4>(st + STAGE, MT_PA, s_d[ring], 0, cols - c0, vec);
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (wid < 2) {   // passes 0 and 1 side by side
            const float *pa, *pd;
            lookup(pa, pd);
            s_a[wid][lane] = pa;
            s_d[wid][lane] = pd;
        }
        __syncthreads();
        if (passes > 0) issue(0, 0);
        at = tt_stacked_next(at, MT_KROWS, M);   // (warp 0: to pass 1)
        int buf = 0, ring = 0;                   // of the current pass
        for (uint64_t left = R; left > 0; left -= min(left, (uint64_t)MT_KROWS)) {
            const int ring1 = ring == 2 ? 0 : ring + 1, ring2 = ring == 0 ? 2 : ring - 1;
            const float *pa = nullptr, *pd = nullptr;
            if (wid == 0) {
                at = tt_stacked_next(at, MT_KROWS, M);
                lookup(pa, pd);
            }
            if (left > MT_KROWS) {
                issue(buf ^ 1, ring1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            if (mtl > 0 && ntl > 0) {
                const float* A = sm + buf * (2 * STAGE) + 32 * wr + g;
                const float* D = sm + buf * (2 * STAGE) + STAGE + 32 * wc + g;
#pragma unroll
                for (int p = 0; p < MT_KROWS / 8; ++p) {
                    if (8 * p >= left) break;
                    const float* Aa = A + (8 * p + t) * MT_PA;
                    const float* Da = D + (8 * p + t) * MT_PA;
                    tt_quarter_step<WHOLE>(sum, Aa, Aa + 8, Aa + 4 * MT_PA, Aa + 4 * MT_PA + 8, 1, Da, Da + 4 * MT_PA, 1, mtl, ntl);
                }
            }
            if (wid == 0) { s_a[ring2][lane] = pa; s_d[ring2][lane] = pd; }   // the ring slot of the pass before
            __syncthreads();
            buf ^= 1;
            ring = ring1;
        }
        float* const dst = td.grad[kc] + (size_t)ik * td.slice_floats[kc];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int a = a0 + 32 * wr + 16 * mt + 8 * h + g, c = c0 + 32 * wc + 8 * nt + 2 * t;
                    if (a >= ra || c >= cols) continue;
                    float* d = dst + (size_t)a * cols + c;
                    if (vec) *reinterpret_cast<float2*>(d) = make_float2(sum[mt][nt][2 * h], sum[mt][nt][2 * h + 1]);
                    else {
                        d[0] = sum[mt][nt][2 * h];
                        if (c + 1 < cols) d[1] = sum[mt][nt][2 * h + 1];
                    }
                }
        if constexpr (FOLD) {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) sum[mt][nt][i] = 0.f;
        } else {
            return;
        }
    }

    // ---------------------------------------------------------------------------------- tiles of Y
    __shared__ const float* s_row[MT_EDGE];    // dP row of each stacked row
    __shared__ const float* s_core[MT_EDGE];   // row of the slice for each a
    __shared__ float* s_out[MT_EDGE];
    const uint64_t items = (R + MT_EDGE - 1) / MT_EDGE * (uint32_t)ach;   // (one or two of a: r <= 128)
    const int cpasses = (cols + MT_KROWS - 1) / MT_KROWS;
    const uint32_t first = FOLD ? blockIdx.z : blockIdx.z - (uint32_t)dgz, step = (uint32_t)(FOLD ? dgz : yctas);
    for (uint64_t it = first; it < items; it += step) {
        const int a0 = (int)(it & (uint32_t)(ach - 1)) * MT_EDGE;
        const uint64_t row0 = (it >> (ach - 1)) * MT_EDGE;
        if (tid < MT_EDGE) {
            const StackedRow r = tt_stacked_next(tt_stacked_row(row0, M), tid, M);
            const float* pd = nullptr;
            float* py = nullptr;
            if (r.node < j1 - j0) {
                const uint32_t v = w.tnode[k][j0 + r.node];
                pd = w.dP[k] + (size_t)v * w.stride[k] + (size_t)r.m * cols;
                py = w.Y[k] + (size_t)v * w.stride[k - 1] + (size_t)r.m * ra;
            }
            s_row[tid] = pd;
            s_out[tid] = py;
        } else {
            const int a = a0 + tid - MT_EDGE;
            s_core[tid - MT_EDGE] = a < ra ? td.core[kc] + (size_t)ik * td.slice_floats[kc] + (size_t)a * cols : nullptr;
        }
        __syncthreads();
        const int mtl = min(2, max(0, ((int)min(R - row0, (uint64_t)MT_EDGE) - 32 * wr + 15) / 16));
        const int ntl = min(4, max(0, (ra - a0 - 32 * wc + 7) / 8));
        auto issue = [&](int c) {
            float* st = sm + (c & 1) * (2 * STAGE);
            const int off = c * MT_KROWS, avail = cols - off;
            tt_stage_rows<MT_EDGE, MT_KROWS / 4>(st, MT_PC, s_row, off, avail, vec);
            tt_stage_rows<MT_EDGE, MT_KROWS / 4>(st + STAGE, MT_PC, s_core, off, avail, vec);
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        issue(0);
        for (int c = 0; c < cpasses; ++c) {
            if (c + 1 < cpasses) {
                issue(c + 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            if (mtl > 0 && ntl > 0) {
                const float* D = sm + (c & 1) * (2 * STAGE) + (32 * wr + g) * MT_PC + t;
                const float* B = sm + (c & 1) * (2 * STAGE) + STAGE + (32 * wc + g) * MT_PC + t;
#pragma unroll
                for (int p = 0; p < MT_KROWS / 8; ++p) {
                    if (c * MT_KROWS + 8 * p >= cols) break;
                    const float* Da = D + 8 * p;
                    const float* Ba = B + 8 * p;
                    tt_quarter_step<WHOLE>(sum, Da, Da + 8 * MT_PC, Da + 4, Da + 8 * MT_PC + 4, MT_PC, Ba, Ba + 4, MT_PC, mtl, ntl);
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float* out = s_out[32 * wr + 16 * mt + 8 * h + g];
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    const int a = a0 + 32 * wc + 8 * nt + 2 * t;
                    if (out && a < ra) {
                        if (vec) *reinterpret_cast<float2*>(out + a) = make_float2(sum[mt][nt][2 * h], sum[mt][nt][2 * h + 1]);
                        else {
                            out[a] = sum[mt][nt][2 * h];
                            if (a + 1 < ra) out[a + 1] = sum[mt][nt][2 * h + 1];
                        }
                    }
                    sum[mt][nt][2 * h] = 0.f;
                    sum[mt][nt][2 * h + 1] = 0.f;
                }
            }
        __syncthreads();   // the addresses are rewritten for the next tile
    }
}

// dP_{k-1}[parent] (k = 2: the first core's gradient slice) = sum of the Y rows of the parent's children, which are
// contiguous in sorted order.  One warp per parent and block of 32 float4 (or 32 floats where a row is no multiple of four
// floats); where there are no more of these than CTAs, as with the few parents of many children at k = 2, the eight warps of
// a CTA share one.  Rows narrower than 32 pieces
// put several children side by side, and eight children per lane are in flight at a time, the last ones included (a loop
// over the remainder would make a round trip for each).  Bound by the latency of those round trips where there are few
// parents: 331 parents of 112 children (16 floats) took 31 us with one warp per parent and one
// child at a time, 7 us now; bound by HBM on large batches (0.7 GB of Y in 90 us).
template <bool VEC>
__device__ __forceinline__ void tt_mid_sum_item(const WsView& w, const TableDesc& td, int k, uint32_t pn, uint32_t f0, float4 (*s_sum)[32], int share, int shares)
{
    constexpr int NF = 8;
    using piece_t = typename std::conditional<VEC, float4, float>::type;
    constexpr uint32_t PF = VEC ? 4 : 1;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t pitch = (uint32_t)w.stride[k - 1] / PF, np = (uint32_t)(td.P[k - 1] * td.r[k - 1]) / PF;
    const uint32_t c0 = w.cstart[k - 1][pn], n = w.cstart[k - 1][pn + 1] - c0;
    uint32_t lpr = 32;
    while (lpr > 1 && lpr / 2 >= np) lpr >>= 1;
    const uint32_t slots = 32u / lpr, slot = lane / lpr, f = f0 + lane % lpr;
    const piece_t* y = reinterpret_cast<const piece_t*>(w.Y[k]) + (size_t)c0 * pitch + f;
    RowAcc<VEC, 1> s;
    s.clear();
    if (f < np)
        for (uint32_t v0 = slot + slots * (uint32_t)share; v0 < n; v0 += NF * slots * (uint32_t)shares) {
            piece_t x[NF];
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const uint32_t v = v0 + (uint32_t)i * slots * (uint32_t)shares;
                x[i] = v < n ? __ldg(y + (size_t)v * pitch) : piece_t{};
            }
#pragma unroll
            for (int i = 0; i < NF; ++i) s.add_shared(&x[i]);
        }
    for (uint32_t o = lpr; o < 32; o <<= 1)
#pragma unroll
        for (uint32_t i = 0; i < PF; ++i) s.v[i] += __shfl_xor_sync(0xffffffffu, s.v[i], o);
    if (shares > 1) {   // the warps of the CTA, in order
        s.store(reinterpret_cast<float*>(&s_sum[share][lane]), (int)PF, 0);
        __syncthreads();
        if (share == 0)
            for (int i = 1; i < shares; ++i) s.add_shared(&s_sum[i][lane]);
        __syncthreads();
        if (share != 0) return;
    }
    if (f >= np || slot != 0) return;
    float* dst = (k == 2 ? td.grad[0] + (size_t)w.val[1][pn] * td.slice_floats[0] : w.dP[k - 1] + (size_t)pn * w.stride[k - 1]) + PF * f;
    s.store(dst, (int)PF, 0);
    if (k == 2 && w.fused_lr != 0.f) {   // the slices of present first digits are final here: the fused update goes with them
        float* c = td.core[0] + (size_t)w.val[1][pn] * td.slice_floats[0] + PF * f;
        RowAcc<VEC, 1> u;
#pragma unroll
        for (uint32_t i = 0; i < PF; ++i) u.v[i] = c[i] - w.fused_lr * s.v[i];
        u.store(c, (int)PF, 0);
    }
}

// blocks: of 32 pieces, in the widest row of level k - 1
__global__ void __launch_bounds__(256) k_mid_sum(WsView w, int k, uint32_t blocks)
{
    tt_pdl_enter();
    __shared__ float4 s_sum[8][32];
    const int wid = threadIdx.x >> 5;
    const uint64_t items = (uint64_t)w.counters[CTR_LEVEL0 + k - 1] * blocks;
    const int shares = items <= gridDim.x ? 8 : 1;
    const uint64_t first = shares > 1 ? blockIdx.x : (uint64_t)blockIdx.x * 8 + wid, step = (uint64_t)gridDim.x * (8 / shares);
    for (uint64_t it = first; it < items; it += step) {
        const uint32_t pn = (uint32_t)(it / blocks), f0 = (uint32_t)(it % blocks) * 32u;
        const TableDesc& td = w.tdesc[tt_find_table(w.tb[k - 1], w.T, pn)];
        const uint32_t nout = (uint32_t)(td.P[k - 1] * td.r[k - 1]);
        if (nout & 3) {   // the first core's slices are not 16-byte aligned
            if (f0 < nout) tt_mid_sum_item<false>(w, td, k, pn, f0, s_sum, shares > 1 ? wid : 0, shares);
        } else if (4 * f0 < nout) tt_mid_sum_item<true>(w, td, k, pn, f0, s_sum, shares > 1 ? wid : 0, shares);
    }
}

template <int M, int RA, int COLS>
static cudaError_t tt_launch_mid(dim3 grid, cudaStream_t st, const WsView& w, int k, int variant, int lbase)
{
    constexpr size_t smem = tt_mid_smem_bytes<M, RA, COLS>();
    cudaError_t e = cudaFuncSetAttribute(k_mid_mma<M, RA, COLS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return tt_launch_pdl(k_mid_mma<M, RA, COLS>, grid, dim3(128), smem, st, w, k, variant, lbase);
}

cudaError_t tt_launch_bwd_middle(tt_emb* h, cudaStream_t s)
{
    WsView& w = h->v;
    cudaError_t e;
    for (int k = h->K - 1; k >= 2; --k) {
        bool any_fast[TT_NUM_MIDFAST] = {};
        uint32_t sum_blocks = 1;
        int dgz = 1;                  // generic shapes: tiles of the slice gradient,
        int64_t ytiles = 1;           // most tiles of Y of a slice
        bool whole = true;            // all shapes fill the quarters of their tiles
        for (int t = 0; t < h->T; ++t) {
            const TableDesc& td = h->tab[t];
            const int kc = k - 1;
            const uint32_t nout = (uint32_t)(td.P[kc] * td.r[kc]), pieces = (nout & 3) ? nout : nout / 4;
            if ((pieces + 31) / 32 > sum_blocks) sum_blocks = (pieces + 31) / 32;
            if (td.midfast[k] >= 0) { any_fast[td.midfast[k]] = true; continue; }
            if (td.r[kc] % (MT_EDGE / 2) != 0 || td.d[kc] * td.r[kc + 1] % (MT_EDGE / 2) != 0) whole = false;
            const int tiles = ((td.r[kc] + MT_EDGE - 1) / MT_EDGE) * ((td.d[kc] * td.r[kc + 1] + MT_EDGE - 1) / MT_EDGE);
            if (tiles > dgz) dgz = tiles;
            const int64_t rows = (int64_t)(td.prefix_space[k - 1] < w.cap[k] ? td.prefix_space[k - 1] : w.cap[k]) * td.P[kc];
            const int64_t yt = (rows + MT_EDGE - 1) / MT_EDGE * ((td.r[kc] + MT_EDGE - 1) / MT_EDGE);
            if (yt > ytiles) ytiles = yt;
        }
        const int ngen = h->mcount[k][0];
        // level K-1's digit-major list already exists: the forward built it to order its sweep
        if (k != h->K - 1 && (e = h->serial ? tt_launch_tlist(h, k, s) : tt_join(h, s, 1)) != cudaSuccess) return e;
        // the shape variants are independent (different tables): run them side by side so that the tail of one
        // (a few long node lists) overlaps the others
        int nfast = 0;
        for (int v = 0; v < TT_NUM_MIDFAST; ++v) nfast += any_fast[v] ? 1 : 0;
        const bool fork = nfast + (ngen > 0 ? 1 : 0) > 1 && !h->serial;
        if (fork && (e = tt_fork(h, s, 4)) != cudaSuccess) return e;
        int slot = 0;
        auto st = [&]() { return fork ? h->side[(slot++) & 3] : s; };
        // grid of variant v: its own tables only, slices up to the largest n_k among them
        auto mgrid = [&](int v) { return dim3(h->mmaxn[k][v + 1], h->mcount[k][v + 1]); };
        auto mlist = [&](int v) { return (2 + k) * h->T + h->mbase[k][v + 1]; };
        if (any_fast[0]) { if ((e = tt_launch_mid<4, 32, 128>(mgrid(0), st(), w, k, 0, mlist(0))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[1]) { if ((e = tt_launch_mid<4, 16, 128>(mgrid(1), st(), w, k, 1, mlist(1))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[2]) { if ((e = tt_launch_mid<4, 32, 64>(mgrid(2), st(), w, k, 2, mlist(2))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[3]) { if ((e = tt_launch_mid<4, 16, 64>(mgrid(3), st(), w, k, 3, mlist(3))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[4]) { if ((e = tt_launch_mid<2, 32, 128>(mgrid(4), st(), w, k, 4, mlist(4))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[5]) { if ((e = tt_launch_mid<2, 16, 64>(mgrid(5), st(), w, k, 5, mlist(5))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[6]) { if ((e = tt_launch_mid<2, 32, 64>(mgrid(6), st(), w, k, 6, mlist(6))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[7]) { if ((e = tt_launch_mid<2, 16, 32>(mgrid(7), st(), w, k, 7, mlist(7))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[8]) { if ((e = tt_launch_mid<4, 8, 32>(mgrid(8), st(), w, k, 8, mlist(8))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[9]) { if ((e = tt_launch_mid<2, 8, 32>(mgrid(9), st(), w, k, 9, mlist(9))) != cudaSuccess) return e; tt_note_launch(); }
        if (any_fast[10]) { if ((e = tt_launch_mid<2, 8, 16>(mgrid(10), st(), w, k, 10, mlist(10))) != cudaSuccess) return e; tt_note_launch(); }
        if (ngen > 0) {
            // very many slices fill the chip with their dG tiles, and most of them have no or few nodes: no CTAs of their own for Y
            const int64_t slices = (int64_t)h->mmaxn[k][0] * ngen;
            const bool fold = slices >= 64 * h->sm_count;
            const int yctas = fold ? 0 : tt_ctas_per_slice(h->sm_count, slices, ytiles);
            auto kern = whole ? (fold ? k_mid_tile<true, true> : k_mid_tile<false, true>) : (fold ? k_mid_tile<true, false> : k_mid_tile<false, false>);
            if ((e = tt_launch_pdl(kern, dim3(h->mmaxn[k][0], ngen, dgz + yctas), dim3(128), 0, st(), w, k, mlist(-1), dgz, yctas)) != cudaSuccess) return e;
            tt_note_launch();
        }
        if (fork && (e = tt_join(h, s, 4)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(k_mid_sum, dim3(h->sm_count * 8), dim3(256), 0, s, w, k, sum_blocks)) != cudaSuccess) return e;
        tt_note_launch();
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- SGD

__global__ void __launch_bounds__(256) k_sgd(WsView w, float lr, int only_unfused)
{
    tt_pdl_enter();
    const int t = blockIdx.y / w.K, k = blockIdx.y % w.K;
    const TableDesc& td = w.tdesc[t];
    if (only_unfused && ((td.sgd_mask >> k) & 1)) return;   // updated by the kernel that finalised its gradient
    float* __restrict__ G = td.core[k];
    const float* __restrict__ dG = td.grad[k];
    const int64_t n = td.core_floats[k];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        G[i] = G[i] - lr * dG[i];
}

cudaError_t tt_launch_sgd(tt_emb* h, float lr, bool only_unfused, cudaStream_t s)
{
    k_sgd<<<dim3(64, h->T * h->K), 256, 0, s>>>(h->v, lr, only_unfused ? 1 : 0);
    tt_note_launch();
    return cudaGetLastError();
}
