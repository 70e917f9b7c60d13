// Grouping and schedule in one kernel, where the bitmaps are short (tt_use_cluster): one cluster of sixteen CTAs runs every
// step, with the cluster's hardware barrier between the steps.
//
// The steps of grouping.cu are a chain of fifteen dependent kernels (marks, a scan per level, links, the digit-major list,
// costs, boundaries), 3 to 5 us each however little they do.  Sixteen SMs do the same work on a few thousand lookups in
// less than the launches cost: 1 k lookups, one table, grouping and schedule 74 -> 33 us, now bound by the latency of the
// dependent loads in each step (one to three L2 round trips between two barriers).  The step functions are those of
// group.cuh; only the distribution over threads differs.
// Where every table is swept by warps that take one batch of groups at a time, the units hold equal group counts instead of
// equal costs, whatever the batch, and the costs and their scan are left out.  Whole forward calls with equal counts / equal costs
// (4x4x4, rank 16), us: 1 table, 11 k lookups 55 / 67, 0.5 M 136 / 147, 10 M 743 / 773; 8 tables of 10 M rows, 4 M lookups 811 / 860;
// the other way only for few lookups of large tables whose popular prefixes hold hundreds of rows (1 table of 40 M rows, 11 k
// lookups, popular rows first 107 / 97; 2 tables 127 / 118).
// The cluster needs sixteen SMs of one GPC at one moment.  Calls of 1 k lookups beside another stream's kernels, cluster / a
// kernel per step, us: idle GPU 47 / 77; copies of 1 GB, median of the calls that meet them 0.66 / 2.2 ms (each kernel of the
// chain waits for its turn); matrix products 0.72 / 0.70 ms; forwards of 16 tables 0.11 / 0.84 ms.
#include "common.cuh"
#include "scan.cuh"
#include "group.cuh"

#define GC_THREADS 1024
#define GC_CTAS 16
#define GC_NODES 4     // nodes that a thread links at a time

// all writes of the cluster's threads before the barrier are visible to all of them after it
__device__ __forceinline__ void gc_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// elements that each CTA takes
__device__ __forceinline__ uint32_t gc_run(uint32_t n) { return (n + GC_CTAS - 1) / GC_CTAS; }

#define GC_IT 4
#define GC_TILE (GC_THREADS * GC_IT)
// Values of one tile of the CTA's run [.., hi): ex holds their exclusive prefixes inside their warps, sm the warps' (element order:
// stripe j, then warp); the tile's sum comes back.
template <class F>
__device__ __forceinline__ uint32_t gc_load(const F& f, uint32_t base, uint32_t hi, int& hint, uint32_t (&v)[GC_IT], uint32_t (&ex)[GC_IT],
                                            int (&at)[GC_IT], uint32_t* sm)
{
    const uint32_t tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int j = 0; j < GC_IT; ++j) {
        const uint32_t i = base + (uint32_t)j * GC_THREADS + tid;
        v[j] = 0;
        if (i < hi) {
            hint = f.locate_from(i, hint);
            v[j] = f.value(i, hint);
        }
        at[j] = hint;
    }
    __syncthreads();        // the warps' sums of the tile (or scan) before are read
#pragma unroll
    for (int j = 0; j < GC_IT; ++j) {
        const uint32_t a = base + (uint32_t)j * GC_THREADS + tid < hi ? tt_scan_amount(f, v[j], 0) : 0u;
        uint32_t incl = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        ex[j] = incl - a;
        if (lane == 31) sm[j * (GC_THREADS / 32) + wid] = incl;
    }
    __syncthreads();
    if (wid == 0) {   // exclusive scan of the warps' sums, GC_IT per lane
        uint32_t x[GC_IT], s = 0;
#pragma unroll
        for (int j = 0; j < GC_IT; ++j) { x[j] = sm[lane * GC_IT + j]; s += x[j]; }
        uint32_t incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t run = incl - s;
#pragma unroll
        for (int j = 0; j < GC_IT; ++j) { sm[lane * GC_IT + j] = run; run += x[j]; }
        if (lane == 31) sm[GC_THREADS / 32 * GC_IT] = run;
    }
    __syncthreads();
    return sm[GC_THREADS / 32 * GC_IT];
}
template <class F>
__device__ __forceinline__ void gc_store(const F& f, uint32_t base, uint32_t hi, uint32_t carry, const uint32_t (&v)[GC_IT], const uint32_t (&ex)[GC_IT],
                                         const int (&at)[GC_IT], const uint32_t* sm)
{
#pragma unroll
    for (int j = 0; j < GC_IT; ++j) {
        const uint32_t i = base + (uint32_t)j * GC_THREADS + threadIdx.x;
        if (i < hi) f.emit(i, carry + sm[j * (GC_THREADS / 32) + (threadIdx.x >> 5)] + ex[j], v[j], at[j]);
    }
}
// this CTA's sum into the shared memory of all sixteen, by their first GC_CTAS threads (or those of a warp)
__device__ __forceinline__ void gc_tell(uint32_t* sums, uint32_t tot, uint32_t thread)
{
    if (thread < GC_CTAS) {
        uint32_t remote;
        const uint32_t local = (uint32_t)__cvta_generic_to_shared(sums + blockIdx.x);
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(thread));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(tot) : "memory");
    }
}
// sum of the CTAs before this one; the first CTA reports that of all
template <class F>
__device__ __forceinline__ uint32_t gc_carry(const F& f, const uint32_t* sums)
{
    uint32_t carry = 0, all = 0;
#pragma unroll
    for (uint32_t i = 0; i < GC_CTAS; ++i) {
        const uint32_t x = sums[i];
        carry += i < blockIdx.x ? x : 0u;
        all += x;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) f.total(all);
    return carry;
}

// Exclusive scan of f over n elements: every CTA takes a run of them.  The CTAs' sums go straight into the shared memory of
// all sixteen (`sums`, a slot of its own for every scan of the kernel); a run of up to GC_TILE elements stays in registers
// between the sum and the second pass.  One barrier inside, none at the end.
template <class F>
__device__ __forceinline__ void gc_scan(const F& f, uint32_t n, uint32_t* sums, uint32_t* sm)
{
    const uint32_t per = gc_run(n), lo = min(n, blockIdx.x * per), hi = min(n, lo + per);
    int hint = lo < hi ? f.locate(lo) : 0;
    uint32_t v[GC_IT], ex[GC_IT], tot = 0;
    int at[GC_IT];
    const bool one = per <= GC_TILE;
    if (one) tot = gc_load(f, lo, hi, hint, v, ex, at, sm);
    else {
        uint32_t amount = 0;
        for (uint32_t i = lo + threadIdx.x; i < hi; i += GC_THREADS) amount += tt_scan_amount(f, f.value(i, hint), 0);
        tt_block_excl_scan(amount, sm, tot);
    }
    gc_tell(sums, tot, threadIdx.x);
    gc_sync();
    uint32_t carry = gc_carry(f, sums);
    if (one) gc_store(f, lo, hi, carry, v, ex, at, sm);
    else
        for (uint32_t base = lo; base < hi; base += GC_TILE) {
            hint = base == lo ? f.locate(lo) : hint;
            tot = gc_load(f, base, hi, hint, v, ex, at, sm);
            gc_store(f, base, hi, carry, v, ex, at, sm);
            carry += tot;
        }
}

// The same for several scans at once, with one barrier for all of them (gc_scan pays one or two per scan, and each costs a round
// trip through L2 besides the barrier itself).  First gc_amount for every scan, then gc_exchange, then gc_emit for every scan, whose
// values come from L1 the second time.
template <class F>
__device__ __forceinline__ void gc_amount(const F& f, uint32_t n, uint32_t* warp_sums /* [32] */)
{
    const uint32_t per = gc_run(n), lo = min(n, blockIdx.x * per), hi = min(n, lo + per);
    uint32_t amount = 0;
#pragma unroll 4
    for (uint32_t i = lo + threadIdx.x; i < hi; i += GC_THREADS) amount += tt_scan_amount(f, f.value(i, 0), 0);   // (no functor's value asks for the hint)
    amount = __reduce_add_sync(0xffffffffu, amount);
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = amount;
}
__device__ __forceinline__ void gc_exchange(uint32_t (*warp_sums)[GC_THREADS / 32], uint32_t (*sums)[GC_CTAS], int scans)
{
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (wid < (uint32_t)scans) gc_tell(sums[wid], __reduce_add_sync(0xffffffffu, warp_sums[wid][lane]), lane);
    gc_sync();
}
template <class F>
__device__ __forceinline__ void gc_emit(const F& f, uint32_t n, const uint32_t* sums, uint32_t* sm)
{
    const uint32_t per = gc_run(n), lo = min(n, blockIdx.x * per), hi = min(n, lo + per);
    uint32_t v[GC_IT], ex[GC_IT], carry = gc_carry(f, sums);
    int at[GC_IT], hint = lo < hi ? f.locate(lo) : 0;
    for (uint32_t base = lo; base < hi; base += GC_TILE) {
        const uint32_t tot = gc_load(f, base, hi, hint, v, ex, at, sm);
        gc_store(f, base, hi, carry, v, ex, at, sm);
        carry += tot;
    }
}

// presence bits of the words of level k that this CTA scans, a warp per word, four words at a time; from the level below once it is
// scanned, or (BITS) from its bits, and then with the marks of the digit-major order of level K-1
template <bool BITS>
__device__ __forceinline__ void gc_level_bits(const WsView& w, int k, bool mark)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t n = w.total_words_l[k], per = gc_run(n), lo = min(n, blockIdx.x * per), hi = min(n, lo + per);
    const LevelScan<const WsView&> ls{w, k};
    int t = lo < hi ? ls.locate(lo) : 0;
    for (uint32_t i0 = lo + wid; i0 < hi; i0 += GC_THREADS / 32 * 4) {
        bool present[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t i = i0 + (uint32_t)j * (GC_THREADS / 32);
            present[j] = false;
            if (i < hi) {
                t = ls.locate_from(i, t);
                const TableDesc& td = w.tdesc[t];
                const uint32_t p = ((i - td.lword_base[k]) << 5) + lane;
                present[j] = BITS ? tt_prefix_any(w, td, k, p) : tt_prefix_present(w, td, k, p);
                if (mark && present[j]) tt_tmark_value(w, td, k, p);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t i = i0 + (uint32_t)j * (GC_THREADS / 32);
            const unsigned bits = __ballot_sync(0xffffffffu, present[j]);
            if (lane == 0 && i < hi) w.bml[k][i] = make_uint2(bits, 0u);
        }
    }
}


// rows: from the row ids on (workspace regions cleared here); otherwise the row bitmap is scanned already
// BITS: all bitmaps are written before any of them is scanned, and all are scanned at once; level: one more than the highest level
// whose bitmap this kernel writes from the bits of the level below; links: 0 ends after the scans (BITS).  !BITS (level = 0; a radix is past TT_BITS_RADIX): level by level,
// each from the ranks of the one below.  (One kernel for both was longer for each: two tables, two cores, 4.7 k lookups, call 89 us,
// 85 apart.)
template <bool BITS>
__global__ void __launch_bounds__(GC_THREADS) k_group_cluster(const __grid_constant__ WsView w, int rows, int level, int links)
{
    tt_pdl_enter();
    __shared__ uint32_t sm[GC_THREADS / 32 * GC_IT + 1];
    __shared__ uint32_t sums[TT_MAXK + 1][GC_CTAS];   // a slot for every scan; [0]: of the digit-major bitmap, [K]: of the costs, where these are scanned late
    const int K = w.K;
    const uint32_t tid = threadIdx.x, first = blockIdx.x * GC_THREADS + tid, step = GC_CTAS * GC_THREADS;
    const bool digit_major = tt_digit_major(w);
    if (rows) {
        if (first < 16 + 64) reinterpret_cast<uint32_t*>(w.status)[first] = 0u;   // status and counters are adjacent
        uint4* bm4 = reinterpret_cast<uint4*>(w.bm);                             // a whole number of scan tiles
        for (uint32_t i = first; i < w.total_words / 2; i += step) bm4[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (digit_major && (rows || !BITS))   // (otherwise k_mark has cleared it)
        for (uint32_t i = first; i < w.ttotal_words[K - 1]; i += step) w.tbm[K - 1][i] = make_uint2(0u, 0u);
    gc_sync();   // also: every CTA runs before another writes into its shared memory
    if (rows) {
        tt_check_offsets<false>(w, first, step);
        tt_clear_pairs(w);
        tt_mark_rows<false>(w, first, step, (int64_t)step * 4);
        gc_sync();
    }
    const uint32_t twords = digit_major ? w.ttotal_words[K - 1] : 0u;
    bool listed = BITS;     // the digit-major bitmap is marked and scanned
    if constexpr (BITS) {
        __shared__ uint32_t warp_sums[TT_MAXK + 1][GC_THREADS / 32];
        for (int k = level - 1; k >= 1; --k) {
            gc_level_bits<true>(w, k, digit_major && k == K - 1);
            if (k > 1) gc_sync();
            else __syncthreads();   // the words of level 1 are scanned by the CTA that has written them
        }
        // scans 0 .. K - 2: levels 1 .. K - 1; K - 1: the digit-major bitmap; K: the rows
        const PopScan<TT_SCAN_TILE, const WsView&> ps{w};
        const TPopScan<const WsView&> ts{w, K - 1};
        for (int k = 1; k < K; ++k) gc_amount(LevelScan<const WsView&>{w, k}, w.total_words_l[k], warp_sums[k - 1]);
        gc_amount(ts, twords, warp_sums[K - 1]);
        gc_amount(ps, rows ? w.total_words : 0u, warp_sums[K]);
        gc_exchange(warp_sums, sums, K + 1);
        if (rows) gc_emit(ps, w.total_words, sums[K], sm);
        for (int k = 1; k < K; ++k) gc_emit(LevelScan<const WsView&>{w, k}, w.total_words_l[k], sums[k - 1], sm);
        if (digit_major) gc_emit(ts, twords, sums[K - 1], sm);
        if (!links) return;
        gc_sync();
        if (digit_major) {   // more nodes than there is room for: the marks are those of the nodes that are kept
            uint32_t all = 0;
            for (int i = 0; i < GC_CTAS; ++i) all += sums[K - 2][i];
            if (all > w.cap[K - 1]) {
                listed = false;
                for (uint32_t i = first; i < twords; i += step) w.tbm[K - 1][i] = make_uint2(0u, 0u);
                gc_sync();
            }
        }
    } else {
        if (rows) {
            gc_scan(PopScan<TT_SCAN_TILE, const WsView&>{w}, w.total_words, sums[K], sm);
            gc_sync();
        }
        for (int k = K - 1; k >= 1; --k) {
            gc_level_bits<false>(w, k, false);
            __syncthreads();
            gc_scan(LevelScan<const WsView&>{w, k}, w.total_words_l[k], sums[k], sm);
            gc_sync();
        }
    }
    // links of all levels, a level at a time, and the digit-major list; unit boundaries by the threads that come last
    if (first < (uint32_t)(K - 1)) tt_link_end(w, (int)first + 1);
    for (int k = K - 1; k >= 1; --k) {
        const uint32_t count = w.counters[CTR_LEVEL0 + k];
        const bool top = digit_major && k == K - 1, fill = top && listed && w.equal_units;
        int t = 0;
        for (uint32_t v0 = first; v0 < count; v0 += GC_NODES * step) {   // GC_NODES nodes at a time: their look-ups overlap
            uint32_t val[GC_NODES], at[GC_NODES], up[GC_NODES], rank[GC_NODES];
#pragma unroll
            for (int j = 0; j < GC_NODES; ++j) val[j] = v0 + j * step < count ? w.val[k][v0 + j * step] : 0u;
#pragma unroll
            for (int j = 0; j < GC_NODES; ++j) {
                const uint32_t v = v0 + j * step;
                if (v >= count) break;
                t = j == 0 ? tt_find_table(w.tb[k], w.T, v) : tt_find_table_from(w.tb[k], w.T, v, t);
                const TableDesc& td = w.tdesc[t];
                at[j] = tt_rank_at(w, td, k + 1, val[j] * (uint32_t)td.n[k]);
                if (w.parent[k]) up[j] = tt_rank_at(w, td, k - 1, val[j] / (uint32_t)td.n[k - 1]);
                if (fill) rank[j] = tt_trank(w, td, k, tt_tkey(td, k, val[j]));
                else if (top && !listed) tt_tmark_value(w, td, k, val[j]);
            }
#pragma unroll
            for (int j = 0; j < GC_NODES; ++j) {
                const uint32_t v = v0 + j * step;
                if (v >= count) break;
                w.cstart[k][v] = at[j];
                if (w.parent[k]) w.parent[k][v] = up[j];
                if (fill) w.tnode[k][rank[j]] = v;
            }
        }
    }
    // (from the row ids on, the boundaries are searched for here, where threads are idle: written with the offsets check they took 2 us of
    // every call, 1 k lookups 52 / 50 us)
    if (w.pool_shares > 0 && (rows || tt_pool_bounds_missing(w)))
        for (int64_t ci = step - 1 - first; ci <= w.pool_shares; ci += step) tt_pool_bound(w, ci);
    const int64_t units = (int64_t)w.T * w.units_per_table;
    if (w.equal_units)
        for (int64_t u = step - 1 - first; u < units; u += step) tt_unit_bounds(w, (int)u);
    if ((listed || !digit_major) && w.equal_units) return;
    gc_sync();
    const uint32_t groups = w.counters[CTR_LEVEL0 + K - 1];
    if (digit_major) {
        if (!listed) {
            gc_scan(TPopScan<const WsView&>{w, K - 1}, twords, sums[0], sm);
            gc_sync();
        }
        for (uint32_t v = first; v < groups; v += step)
            tt_tfill_node(w, w.tdesc[tt_find_table(w.tb[K - 1], w.T, v)], K - 1, v, !w.equal_units);
    } else if (!w.equal_units) {
        for (uint32_t g = first; g < groups; g += step)
            w.cost[g] = tt_group_cost(w, w.tdesc[tt_find_table(w.tb[K - 1], w.T, g)], g);
    }
    if (w.equal_units) return;
    gc_sync();
    gc_scan(CostScan<const WsView&>{w}, groups, sums[K], sm);
    gc_sync();
    for (int64_t u = first; u < units; u += step) tt_unit_bounds(w, (int)u);
}

cudaError_t tt_launch_group_cluster(tt_emb* h, bool rows, int level, bool links, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(GC_CTAS);
    cfg.blockDim = dim3(GC_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = GC_CTAS;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, level != 0 ? k_group_cluster<true> : k_group_cluster<false>, h->v, rows ? 1 : 0, level, links ? 1 : 0);
    if (e == cudaSuccess) tt_note_launch();
    return e;
}

// whether the device takes the cluster (sixteen CTAs are past the portable eight): asked once per handle
int tt_group_cluster_ok()
{
    if (cudaFuncSetAttribute(k_group_cluster<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k_group_cluster<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) { cudaGetLastError(); return 0; }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(GC_CTAS);
    cfg.blockDim = dim3(GC_THREADS);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = GC_CTAS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;      // (of the one with more shared memory; the registers are those of 1024 threads either way)
    if (cudaOccupancyMaxActiveClusters(&n, k_group_cluster<true>, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n > 0;
}
