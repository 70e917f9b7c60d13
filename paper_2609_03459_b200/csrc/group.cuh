// Device functions of the grouping and of the schedule, one element (lookup, bitmap word, node, share) at a time, shared by
// the kernels that run each step over the whole chip (grouping.cu) and by the one that runs all steps in one cluster
// (group_cluster.cu).
// The scan functors hold the workspace view by value where a kernel gets the functor as its parameter, by reference inside
// a kernel that has the view.
#pragma once
#include "common.cuh"
#include "scan.cuh"

// ---- shares of the pooling pass

// Share ci starts with the first bag whose offset is >= L ci / C.  The pass that checks the offsets writes the boundaries as
// it goes: bag i + 1 is the first bag of every share whose target lies in (offsets[i], offsets[i + 1]].  (A bisection of
// the offsets per share, 15 dependent loads each, took 6 us of its step in the cluster: 8 tables, 33 k bags, 33 k shares, call
// 652 -> 646 us.  With many bags per share the search is cheaper than two quotients per bag: 60 k shares of 2 M bags grouping and
// schedule 811 / 806 us, of 7.9 M bags 1024 / 1052.  Where one cluster does everything, it searches: k_group_cluster.)

#define TT_POOL_BAGS_PER_SHARE 64
__device__ __forceinline__ bool tt_pool_bounds_by_bag(const WsView& w)
{
    return w.pool_shares > 0 && w.L > 0 && (int64_t)w.T * w.B <= TT_POOL_BAGS_PER_SHARE * w.pool_shares;
}

// first share whose target is past lookup x: the smallest ci with L ci >= C (x + 1).  C (x + 1) < 2^48 is exact in fp64, the
// quotient is off by one at most
__device__ __forceinline__ int64_t tt_first_share(const WsView& w, int64_t x, double invL)
{
    const int64_t num = w.pool_shares * (x + 1);
    int64_t ci = (int64_t)((double)num * invL);
    if (ci * w.L < num) ++ci;
    else if (ci > 0 && (ci - 1) * w.L >= num) --ci;
    return ci;
}
// the shares that start after bag i, 0 <= o = offsets[i] <= o_next = offsets[i + 1] <= L
__device__ __forceinline__ void tt_pool_bounds_after(const WsView& w, int64_t i, int64_t o, int64_t o_next, double invL)
{
    const int64_t C = w.pool_shares, nb = (int64_t)w.T * w.B;
    const int64_t c0 = tt_first_share(w, o, invL), c1 = i + 1 < nb ? tt_first_share(w, o_next, invL) : C;
    for (int64_t ci = c0; ci < c1 && ci < C; ++ci) w.pool_bounds[ci] = i + 1;
    if (i == 0)
        for (int64_t ci = 0; ci < c0 && ci < C; ++ci) w.pool_bounds[ci] = 0;
    if (i + 1 == nb) w.pool_bounds[C] = nb;
}
// otherwise, and with offsets that the check has flagged, the boundaries come from a search: the same one for both neighbours
// of a boundary, so that the shares have no gaps whatever the offsets hold
__device__ __forceinline__ bool tt_pool_bounds_missing(const WsView& w)
{
    return w.pool_shares > 0 && (!tt_pool_bounds_by_bag(w) || (__ldcg(w.status) & TT_EMB_STATUS_OFFSETS));
}
__device__ __forceinline__ void tt_pool_bound(const WsView& w, int64_t ci)
{
    const int64_t C = w.pool_shares, nb = (int64_t)w.T * w.B;
    const int64_t target = (w.L * ci) / C;
    int64_t lo = 0, hi = nb;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(w.offsets + mid) < target) lo = mid + 1; else hi = mid;
    }
    w.pool_bounds[ci] = ci == 0 ? 0 : (ci == C ? nb : lo);
}

// ---- ingest

// first lookup of table t, from the offsets (clamped: malformed ones set a status bit and are used as they are otherwise)
__device__ __forceinline__ int64_t tt_table_start(const WsView& w, int t)
{
    const int64_t o = __ldg(w.offsets + (int64_t)t * w.B);
    return o < 0 ? 0 : (o > w.L ? w.L : o);
}

// Lookups that may be in no bag, before the first offset and from the last one on, have no pair for the backward (what a call before
// left in their place would be counted with rows and bags that this call may not have).  By the grid's first warp: such offsets are an
// error of the caller's.
__device__ __forceinline__ void tt_clear_pairs(const WsView& w)
{
    if (blockIdx.x != 0 || threadIdx.x >= 32 || !w.upairs) return;
    const uint32_t L = (uint32_t)w.L;
    auto clampL = [&](int64_t o) { return o < 0 ? 0u : o > w.L ? L : (uint32_t)o; };
    uint32_t o0 = clampL(__ldg(w.offsets)), oL = clampL(__ldg(w.offsets + (int64_t)w.T * w.B));
    if (o0 == 0 && oL == L) return;
    if (o0 > oL) oL = 0u;      // bags that go up again may cover any part
    for (uint32_t l = threadIdx.x; l < L; l += 32)
        if (l < o0 || l >= oL) w.upairs[l] = make_uint2(0xffffffffu, 0u);
}

// the offsets: non-decreasing, from 0 to L; first lookup of every table into tl_start and (SHARES) boundaries of the pooling shares.
// Threads first, first + step, ..
template <bool SHARES>
__device__ __forceinline__ void tt_check_offsets(const WsView& w, int64_t first, int64_t step)
{
    const int64_t nb = (int64_t)w.T * w.B;
    bool bad = false;
    auto check = [&](int64_t i, int64_t o) {
        if (o < 0 || o > w.L) bad = true;
        if (i == 0 && o != 0) bad = true;
        if (i == nb && o != w.L) bad = true;
    };
    if (SHARES && tt_pool_bounds_by_bag(w)) {
        const double invL = 1.0 / (double)w.L;
        for (int64_t i = first; i <= nb; i += step) {
            const int64_t o = __ldg(w.offsets + i), o_next = i < nb ? __ldg(w.offsets + i + 1) : o;
            check(i, o);
            if (o_next < o) bad = true;
            else if (i < nb && o >= 0 && o_next <= w.L) tt_pool_bounds_after(w, i, o, o_next, invL);
        }
    } else {
        for (int64_t i = first; i <= nb; i += step) {
            const int64_t o = __ldg(w.offsets + i);
            check(i, o);
            if (i < nb && __ldg(w.offsets + i + 1) < o) bad = true;
        }
    }
    for (int64_t t = first; t <= w.T; t += step) w.tl_start[t] = tt_table_start(w, (int)t);
    if (bad) atomicOr(w.status, TT_EMB_STATUS_OFFSETS);
}

// one presence bit per looked-up row (TL: k_check_offsets has written tl_start); a thread takes lookups first + j * gap (j < 4), then those `step` further on
template <bool TL>
__device__ __forceinline__ void tt_mark_rows(const WsView& w, int64_t first, int64_t gap, int64_t step)
{
    const int64_t L = w.L;
    int t = 0;
    bool bad = false;
    // the table of the last lookup, kept in registers: lookup range, row count, first presence word
    int64_t l_lo = 0, l_hi = 0, tN = 0;
    uint32_t twb = 0;
    for (int64_t base = first; base < L; base += step) {
        int64_t g[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t l = base + (int64_t)j * gap;
            g[j] = l < L ? tt_index(w, l) : -1;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t l = base + (int64_t)j * gap;
            if (l >= L) continue;
            if (!(l_lo <= l && l < l_hi)) {
                auto start = [&](int i) { return TL ? w.tl_start[i] : tt_table_start(w, i); };
                int lo = 0, hi = w.T;   // largest t whose first lookup is not past l
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (start(mid) <= l) lo = mid; else hi = mid;
                }
                t = lo;
                l_lo = start(t);
                l_hi = start(t + 1);
                tN = w.tdesc[t].N;
                twb = w.tdesc[t].word_base;
            }
            if (g[j] < 0 || g[j] >= tN) { bad = true; continue; }
            const uint32_t row = (uint32_t)g[j];
            unsigned* word = &w.bm[twb + (row >> 5)].x;
            const unsigned m = 1u << (row & 31);
            if (!(__ldca(word) & m)) atomicOr(word, m);   // L1 may hold a stale word: at worst a redundant atomic
        }
    }
    if (bad) atomicOr(w.status, TT_EMB_STATUS_INDEX);
}

// val[excl ..] = v0 + (positions of the set bits of `bits`), clipped at `cap`.  Called by all lanes that emit a word
// (also with bits == 0).  A lane writes the first bits of its own word; a word with more is handed to the whole warp,
// one lane per bit: a densely set word then is one coalesced store instead of 32 stores that each touch another
// sector (a tile of the popular first rows of a table took 80 us against 20 us for a sparse one).  Four such words at a time, so that
// their shuffles overlap, gained 1 to 2 % of a call with many dense words (24 tables, 1 M lookups 253 / 249 us) and lost 2 to 3 % with
// few (12 tables, 78 k lookups 270 / 277; 22 tables, 73 k 159 / 163).
#define EMIT_OWN 8
__device__ __forceinline__ void tt_emit_set_bits(uint32_t* __restrict__ val, uint32_t cap, unsigned bits, uint32_t excl, uint32_t v0)
{
    const unsigned act = __activemask();
    const int lane = threadIdx.x & 31;
    const bool dense = __popc(bits) > EMIT_OWN;
    if (!dense) {
        uint32_t slot = excl;
#pragma unroll
        for (int it = 0; it < EMIT_OWN; ++it)
            if (bits) {
                const int b = __ffs(bits) - 1;
                bits &= bits - 1;
                if (slot < cap) val[slot] = v0 + b;
                ++slot;
            }
    }
    unsigned todo = __ballot_sync(act, dense);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const unsigned wb = __shfl_sync(act, bits, src);
        const uint32_t we = __shfl_sync(act, excl, src);
        const uint32_t wv = __shfl_sync(act, v0, src);
        if ((wb >> lane) & 1u) {
            const uint32_t sl = we + __popc(wb & ((1u << lane) - 1u));
            if (sl < cap) val[sl] = wv + lane;
        }
    }
}

// ---- level K: rows

__device__ __forceinline__ void tt_level_words(const WsView& w, int k, uint32_t warp, uint32_t warps);
// side: CTAs at the end of both grids that write the bitmaps of levels K-1 (first kernel) and K-2 (second) from the bits alone, so that
// these steps run beside the scan on the whole chip instead of after it in the cluster
template <int TILE, class View = WsView>
struct PopScan {
    View w;
    uint32_t side = 0;
    __device__ bool beside(uint32_t cta, uint32_t ctas, bool apply) const
    {
        if (cta + side < ctas) return false;
        const int k = w.K - (apply ? 2 : 1);
        const uint32_t per = TT_SCAN_THREADS / 32, warp = (cta + side - ctas) * per + (threadIdx.x >> 5);
        if (k >= 1) tt_level_words(w, k, warp, side * per);
        return true;
    }
    __device__ uint32_t size() const { return w.total_words; }
    // every table starts on a scan-tile boundary: the table of a tile's first word is the table of all its words
    __device__ int locate(uint32_t i0) const
    {
        int lo = 0, hi = w.T;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (w.tdesc[mid].word_base <= i0) lo = mid; else hi = mid;
        }
        return lo;
    }
    __device__ int locate_from(uint32_t i, int t) const
    {
        while (t + 1 < w.T && w.tdesc[t + 1].word_base <= i) ++t;
        return t;
    }
    __device__ uint32_t value(uint32_t i, int) const { return w.bm[i].x; }
    __device__ uint32_t weight(uint32_t bits) const { return __popc(bits); }
    // The first TT_HEAD_TILES tiles of every table go first (CTAs 0 .. HEAD * T - 1, tile position major), the others
    // follow in ascending order.  With the identity rank-to-row mapping the popular rows are the first rows of a table:
    // those tiles are densely set and emit a hundred times the rows of a tile further down (70 us against 6), and in
    // ascending order the dense tiles of the last tables ran alone at the end of the kernel.
    __device__ uint32_t tile_of(uint32_t cta) const
    {
        constexpr uint32_t PER = TT_SCAN_TILE / TILE;   // the order is that of the long scan's tiles, cut finer
        const uint32_t big = big_tile_of(cta / PER);
        return big == 0xffffffffu ? big : big * PER + cta % PER;
    }
    __device__ uint32_t big_tile_of(uint32_t cta) const
    {
        const uint32_t head = (uint32_t)TT_HEAD_TILES * (uint32_t)w.T;
        if (cta < head) {
            const uint32_t p = cta / (uint32_t)w.T, t = cta % (uint32_t)w.T;
            const TableDesc& td = w.tdesc[t];
            return p < td.num_words / TT_SCAN_TILE ? td.word_base / TT_SCAN_TILE + p : 0xffffffffu;
        }
        const uint32_t m = cta - head;
        if (m >= w.rest_tiles) return 0xffffffffu;
        int lo = 0, hi = w.T;                    // the table whose remaining tiles hold number m
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (w.tdesc[mid].rest_base <= m) lo = mid; else hi = mid;
        }
        return w.tdesc[lo].word_base / TT_SCAN_TILE + TT_HEAD_TILES + (m - w.tdesc[lo].rest_base);
    }
    __device__ void emit(uint32_t i, uint32_t excl, uint32_t bits, int t) const
    {
        w.bm[i].y = excl;
        const int K = w.K;
        const uint32_t wb = w.tdesc[t].word_base;
        if (i == wb) w.tb[K][t] = excl < w.cap[K] ? excl : w.cap[K];
        const uint32_t row0 = (i - wb) << 5;
        tt_emit_set_bits(w.val[K], w.cap[K], bits, excl, row0);
    }
    __device__ void total(uint32_t tot) const
    {
        const int K = w.K;
        if (tot > w.cap[K]) { atomicOr(w.status, TT_EMB_STATUS_OVERFLOW); tot = w.cap[K]; }
        w.counters[CTR_LEVEL0 + K] = tot;
        w.tb[K][w.T] = tot;
    }
};

// ---- prefix levels

// number of level-c nodes before the first one whose value is >= pos (c = K: rows; c < K: length-c prefixes)
__device__ __forceinline__ uint32_t tt_rank_at(const WsView& w, const TableDesc& td, int c, uint32_t pos)
{
    const uint2 e = c == w.K ? w.bm[td.word_base + (pos >> 5)] : w.bml[c][td.lword_base[c] + (pos >> 5)];
    const uint32_t r = e.y + __popc(e.x & ((1u << (pos & 31)) - 1u));
    const uint32_t lim = w.counters[CTR_LEVEL0 + c];
    return r < lim ? r : lim;
}

// number of level-c nodes of all tables before position x of table td (x inside the table's space), from the scanned bitmap
__device__ __forceinline__ uint32_t tt_rank_excl(const WsView& w, const TableDesc& td, int c, uint32_t x)
{
    const uint2 e = c == w.K ? w.bm[td.word_base + (x >> 5)] : w.bml[c][td.lword_base[c] + (x >> 5)];
    return e.y + __popc(e.x & ((1u << (x & 31)) - 1u));
}
// ... up to and including position x
__device__ __forceinline__ uint32_t tt_rank_incl(const WsView& w, const TableDesc& td, int c, uint32_t x)
{
    const uint2 e = c == w.K ? w.bm[td.word_base + (x >> 5)] : w.bml[c][td.lword_base[c] + (x >> 5)];
    return e.y + __popc(e.x & (0xffffffffu >> (31 - (x & 31))));
}

// Whether prefix p of level k < K is present, from the scanned bitmap of level k + 1: some node of that level lies in
// [p n_{k+1}, (p + 1) n_{k+1}).
__device__ __forceinline__ bool tt_prefix_present(const WsView& w, const TableDesc& td, int k, uint32_t p)
{
    const int c = k + 1;
    const uint32_t radix = (uint32_t)td.n[k];                       // radix of digit k + 1
    const uint32_t space_c = c == w.K ? (uint32_t)td.N : td.prefix_space[c];
    const uint64_t lo = (uint64_t)p * radix;
    if (p >= td.prefix_space[k] || lo >= space_c) return false;      // rows past N do not exist
    uint64_t hi = lo + radix;
    if (hi > space_c) hi = space_c;
    return tt_rank_incl(w, td, c, (uint32_t)hi - 1u) != tt_rank_excl(w, td, c, (uint32_t)lo);
}

// ... and from the level's bits alone, before it is scanned: some bit of [p n_{k+1}, (p + 1) n_{k+1}) is set.  One load per word, so
// for radices of up to TT_BITS_RADIX only
#define TT_BITS_RADIX 512
__device__ __forceinline__ bool tt_prefix_any(const WsView& w, const TableDesc& td, int k, uint32_t p)
{
    const int c = k + 1;
    const uint32_t radix = (uint32_t)td.n[k], space_c = c == w.K ? (uint32_t)td.N : td.prefix_space[c];
    const uint64_t lo = (uint64_t)p * radix;
    if (p >= td.prefix_space[k] || lo >= space_c) return false;
    const uint32_t first = (uint32_t)lo, last = (uint32_t)(lo + radix < space_c ? lo + radix : space_c) - 1u;
    const uint2* words = c == w.K ? w.bm + td.word_base : w.bml[c] + td.lword_base[c];
    const uint32_t i0 = first >> 5, i1 = last >> 5;
    uint32_t found = 0;
    for (uint32_t i = i0; i <= i1; i += 4) {
        uint32_t x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = i + j <= i1 ? words[i + j].x : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (i + j == i0) x[j] &= 0xffffffffu << (first & 31);
            if (i + j == i1) x[j] &= 0xffffffffu >> (31 - (last & 31));
            found |= x[j];
        }
    }
    return found != 0;
}

// Level k < K from its own presence bitmap: the ascending distinct prefixes of every table.  The level's bits are set by then: from the
// ranks of level k + 1 once that is scanned (k_prefix_bits, gc_level_bits<false>), or from its bits (tt_level_words,
// gc_level_bits<true>).
template <class View = WsView>
struct LevelScan {
    View w;
    int k;
    __device__ uint32_t size() const { return w.total_words_l[k]; }
    __device__ int locate(uint32_t i0) const
    {
        int lo = 0, hi = w.T;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (w.tdesc[mid].lword_base[k] <= i0) lo = mid; else hi = mid;
        }
        return lo;
    }
    __device__ int locate_from(uint32_t i, int t) const
    {
        while (t + 1 < w.T && w.tdesc[t + 1].lword_base[k] <= i) ++t;
        return t;
    }
    __device__ uint32_t value(uint32_t i, int) const { return w.bml[k][i].x; }
    __device__ uint32_t weight(uint32_t bits) const { return __popc(bits); }
    __device__ void emit(uint32_t i, uint32_t excl, uint32_t bits, int t) const
    {
        w.bml[k][i].y = excl;
        const TableDesc& td = w.tdesc[t];
        const uint32_t wb = td.lword_base[k];
        if (i == wb) w.tb[k][t] = excl < w.cap[k] ? excl : w.cap[k];
        const uint32_t p0 = (i - wb) << 5;
        tt_emit_set_bits(w.val[k], w.cap[k], bits, excl, p0);
    }
    __device__ void total(uint32_t tot) const
    {
        if (tot > w.cap[k]) { atomicOr(w.status, TT_EMB_STATUS_OVERFLOW); tot = w.cap[k]; }
        w.counters[CTR_LEVEL0 + k] = tot;
        w.tb[k][w.T] = tot;
    }
};

// Links of level-k node v (the rank look-ups are random 8-byte loads: kept out of the scan, where one thread would walk
// them one after the other): first child at the level below (k + 1; with the "no prefix reuse" study switch the groups of
// level K-1 are the rows themselves, so level K-2 points at rows), and, for the levels whose left operand is looked up
// through it (3..K-1), the parent at level k-1.
__device__ __forceinline__ void tt_link_node(const WsView& w, const TableDesc& td, int k, uint32_t v)
{
    const int K = w.K;
    const bool rows = (w.ablation & 1) && k == K - 1;          // level k holds one node per row, not per prefix
    const int c = ((w.ablation & 1) && k + 1 == K - 1) ? K : k + 1;
    if (!rows) {
        const uint32_t mult = c == k + 1 ? (uint32_t)td.n[k] : td.suffix[k];   // value of the first possible child
        w.cstart[k][v] = tt_rank_at(w, td, c, w.val[k][v] * mult);
    }
    if (w.parent[k]) {
        const uint32_t up = rows ? w.val[K][v] / td.suffix[k - 1] : w.val[k][v] / (uint32_t)td.n[k - 1];
        w.parent[k][v] = tt_rank_at(w, td, k - 1, up);
    }
}
// ... and the end of the level's list of first children
__device__ __forceinline__ void tt_link_end(const WsView& w, int k)
{
    const bool rows = (w.ablation & 1) && k == w.K - 1;
    const int c = ((w.ablation & 1) && k + 1 == w.K - 1) ? w.K : k + 1;
    if (!rows) w.cstart[k][w.counters[CTR_LEVEL0 + k]] = w.counters[CTR_LEVEL0 + c];
}

// ---- digit-major ("transposed") list of the level-k nodes: a second presence-bitmap sort, keyed by (i_k, parent prefix)
// instead of (parent prefix, i_k); tnode[k][rank] = node

__device__ __forceinline__ uint32_t tt_tkey(const TableDesc& td, int k, uint32_t val)
{
    // digit-major key of a level-k node: i_k * (number of possible parents) + parent prefix value
    const uint32_t nk = (uint32_t)td.n[k - 1];
    return (val % nk) * td.prefix_space[k - 1] + val / nk;
}

__device__ __forceinline__ void tt_tmark_value(const WsView& w, const TableDesc& td, int k, uint32_t val)
{
    const uint32_t key = tt_tkey(td, k, val);
    atomicOr(&w.tbm[k][td.tword_base[k] + (key >> 5)].x, 1u << (key & 31));
}
__device__ __forceinline__ void tt_tmark_node(const WsView& w, const TableDesc& td, int k, uint32_t v) { tt_tmark_value(w, td, k, w.val[k][v]); }

// Presence bitmap of level k from the bits of level k + 1, and the marks of the digit-major order of level K-1, by warps `warp`,
// warp + warps, .. of a kernel that scans level k + 1 or one further down
__device__ __forceinline__ void tt_level_words(const WsView& w, int k, uint32_t warp, uint32_t warps)
{
    const int lane = threadIdx.x & 31;
    const bool mark = k == w.K - 1 && tt_digit_major(w);
    const uint32_t n = w.total_words_l[k];
    for (uint32_t i = warp; i < n; i += warps) {
        int lo = 0, hi = w.T;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (w.tdesc[mid].lword_base[k] <= i) lo = mid; else hi = mid;
        }
        const TableDesc& td = w.tdesc[lo];
        const uint32_t p = ((i - td.lword_base[k]) << 5) + lane;
        const bool present = tt_prefix_any(w, td, k, p);
        if (mark && present) tt_tmark_value(w, td, k, p);
        const unsigned bits = __ballot_sync(0xffffffffu, present);
        if (lane == 0) w.bml[k][i] = make_uint2(bits, 0u);
    }
}

template <class View = WsView>
struct TPopScan {
    View w;
    int k;
    __device__ uint32_t size() const { return w.ttotal_words[k]; }
    __device__ int locate(uint32_t) const { return 0; }
    __device__ int locate_from(uint32_t, int hint) const { return hint; }
    __device__ uint32_t value(uint32_t i, int) const { return __popc(w.tbm[k][i].x); }
    __device__ void emit(uint32_t i, uint32_t excl, uint32_t, int) const { w.tbm[k][i].y = excl; }
    __device__ void total(uint32_t) const {}
};

__device__ __forceinline__ uint32_t tt_trank(const WsView& w, const TableDesc& td, int k, uint32_t key)
{
    const uint2 e = w.tbm[k][td.tword_base[k] + (key >> 5)];
    return e.y + __popc(e.x & ((1u << (key & 31)) - 1u));
}

// costs: level K-1, whose list is the order of the sweeps
__device__ __forceinline__ void tt_tfill_node(const WsView& w, const TableDesc& td, int k, uint32_t v, bool costs)
{
    const uint32_t rank = tt_trank(w, td, k, tt_tkey(td, k, w.val[k][v]));
    w.tnode[k][rank] = v;
    if (costs) w.cost[rank] = tt_group_cost(w, td, v);
}

// ---- schedule

// cost of every group in sweep order -> exclusive prefix sums, in place.  The costs are written by the kernel that fills the
// sweep order (k_tfill; k_costs where the order is the natural one): formed inside the two scan kernels, each cost was
// three dependent look-ups that a thread made sixteen times in a row (20 us per kernel for five thousand groups).
template <class View = WsView>
struct CostScan {
    View w;
    __device__ uint32_t size() const { return w.counters[CTR_LEVEL0 + w.K - 1]; }
    __device__ int locate(uint32_t) const { return 0; }
    __device__ int locate_from(uint32_t, int hint) const { return hint; }
    __device__ uint32_t value(uint32_t j, int) const { return w.cost[j]; }
    __device__ void emit(uint32_t g, uint32_t excl, uint32_t, int) const { w.cost[g] = excl; }
    __device__ void total(uint32_t tot) const
    {
        w.cost[size()] = tot;
        w.counters[CTR_COST_TOTAL] = tot;
    }
};

// group range of work unit u = (table, q)
__device__ __forceinline__ void tt_unit_bounds(const WsView& w, int u)
{
    uint32_t g0, g1;
    tt_unit_range(w, u / w.units_per_table, u % w.units_per_table, g0, g1);
    w.unit_rng[u] = make_uint2(g0, g1);
}
