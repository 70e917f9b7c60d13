// Prefix grouping (paper Sec. 3.3: sort, unique, mixed-radix conversion, run-length encoding), integer only.
//
// B200 design: the sort + unique of a table's row ids is a distribution (counting) sort over the row-id
// domain with one presence bit per row.  The bitmaps of all tables (N_t / 8 bytes each) stay resident in
// the 126 MB L2, so marking costs one L2 access per lookup, and an exclusive scan of the word popcounts
// yields (a) the ascending list of distinct rows, (b) a rank structure {bits, base} that maps any row id
// to its slot with one 8-byte load, so no per-lookup inverse map is ever written.  The prefix levels are
// built the same way: one bit per possible length-k prefix (k < K) in a small bitmap over the prefix space, and a scan of
// its word popcounts yields the ascending distinct prefixes; the first child of a prefix is a rank look-up in the next
// level's bitmap, so the run-length encoding of the sorted rows is never walked.  A prefix is present when the level below
// has a node in its range of children: with a kernel per step the scanned bitmap of that level counts them (two rank
// look-ups per possible prefix, k_prefix_bits), with the cluster its bits are looked at before it is scanned, as long as the range is
// short (group.cuh).  The cost of a prefix level is proportional to the size of its prefix space, not to the
// lookups or the rows.  No kernel waits on another CTA.
#include "common.cuh"
#include "scan.cuh"
#include "group.cuh"

// ---------------------------------------------------------------------------------------------- prologue

__global__ void __launch_bounds__(256) k_check_offsets(WsView w)
{
    tt_pdl_enter();
    tt_clear_pairs(w);
    tt_check_offsets<true>(w, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// FUSED: offsets and row ids in one pass (the marks take the tables' ranges from the offsets themselves); otherwise
// k_check_offsets has run.  The registers of eight CTAs per SM: every lookup is one or two requests and little else.
// Bound by the requests of the lookups that find their bit not set: the lookups of a popular row that are in flight before
// its first mark lands queue up on one word.  So a CTA marks 32 lookups, waits for them and then takes all of its share.  Grouping
// without / with, us: one table, 0.5 M lookups (exponent 1.2, 1 M, 10 M, 40 M rows) 91 / 61, 95 / 63, 102 / 72, spread rows 67 / 47,
// 72 / 52, 87 / 69; 8 tables, 1.6 M lookups 126 / 112; 60 tables, 99 M lookups 816 to 905 / 802 to 814 over runs.  8 / 16 / 64 / 128 lookups instead of
// 32: 102 / 103 / 107 / 115 for 103 us (one table of 16 M rows, 0.5 M lookups).  A second test of the word past L1 before the
// atomic (the copy in L1 is often an old one) costs more than the requests it saves: 8 tables 124 us, 60 tables 950.
#define TT_MARK_SEEDS_FROM (1 << 16)   // 8 k lookups: call 78.5 us with them, 78.0 without
// clear: also clears the digit-major bitmap
template <bool FUSED>
__global__ void __launch_bounds__(256, 8) k_mark(WsView w, int clear)
{
    tt_pdl_enter();
    if (clear)
        for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.ttotal_words[w.K - 1]; i += gridDim.x * blockDim.x) w.tbm[w.K - 1][i] = make_uint2(0u, 0u);
    // one warp's lookups first: the popular rows are marked by then, and the other warps find their bits set
    if (w.L >= TT_MARK_SEEDS_FROM) {
        if (threadIdx.x < 32) tt_mark_rows<!FUSED>(w, (int64_t)blockIdx.x * blockDim.x * 4 + threadIdx.x, w.L, w.L);
        __syncthreads();
    }
    if (FUSED) tt_check_offsets<true>(w, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
    tt_mark_rows<!FUSED>(w, (int64_t)blockIdx.x * blockDim.x * 4 + threadIdx.x, blockDim.x, (int64_t)gridDim.x * blockDim.x * 4);
    if (FUSED) tt_clear_pairs(w);
}

// ---------------------------------------------------------------------------------------------- prefix levels

// Presence bitmap of level k < K (one bit per possible length-k prefix of every table) from level k + 1.  One warp per word,
// one lane per prefix (the two rank look-ups of a prefix are dependent loads: 32 of them one after the other per thread
// took 25 us even for the few words of level 1); the words are written whole (no memset, no atomics).
__global__ void __launch_bounds__(256) k_prefix_bits(WsView w, int k)
{
    tt_pdl_enter();
    const int lane = threadIdx.x & 31;
    const uint32_t nwords = w.total_words_l[k];
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nwords; i += nwarps) {
        int lo_t = 0, hi_t = w.T;
        while (hi_t - lo_t > 1) {
            const int mid = (lo_t + hi_t) >> 1;
            if (w.tdesc[mid].lword_base[k] <= i) lo_t = mid; else hi_t = mid;
        }
        const TableDesc& td = w.tdesc[lo_t];
        const unsigned bits = __ballot_sync(0xffffffffu, tt_prefix_present(w, td, k, ((i - td.lword_base[k]) << 5) + lane));
        if (lane == 0) w.bml[k][i] = make_uint2(bits, 0u);
    }
}

// Links of all levels (blockIdx.y = K - 1 - k), and the marks of the digit-major order of the level-(K-1) nodes (`mark`) or, where it
// is marked and scanned already, its list (`fill`)
__global__ void __launch_bounds__(256) k_links(WsView w, int mark, int fill)
{
    tt_pdl_enter();
    const int k = w.K - 1 - (int)blockIdx.y;
    const uint32_t count = w.counters[CTR_LEVEL0 + k];
    const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x;
    if (first == 0) tt_link_end(w, k);
    for (uint32_t v = first; v < count; v += gridDim.x * blockDim.x) {
        const TableDesc& td = w.tdesc[tt_find_table(w.tb[k], w.T, v)];
        if (mark && blockIdx.y == 0) tt_tmark_node(w, td, k, v);
        if (fill && blockIdx.y == 0) tt_tfill_node(w, td, k, v, false);
        tt_link_node(w, td, k, v);
    }
}

// Study switch "no prefix reuse": every distinct row is a group of its own at level K-1
__global__ void __launch_bounds__(256) k_unique_groups(WsView w)
{
    tt_pdl_enter();
    const int K = w.K, k = K - 1;
    const uint32_t count = w.counters[CTR_LEVEL0 + K] < w.cap[k] ? w.counters[CTR_LEVEL0 + K] : w.cap[k];
    const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x;
    if (first == 0) {
        w.counters[CTR_LEVEL0 + k] = count;
        w.cstart[k][count] = count;
    }
    if (first <= (uint32_t)w.T) w.tb[k][first] = w.tb[K][first] < count ? w.tb[K][first] : count;
    for (uint32_t v = first; v < count; v += gridDim.x * blockDim.x) {
        const int t = tt_find_table(w.tb[K], w.T, v);
        w.val[k][v] = w.val[K][v] / (uint32_t)w.tdesc[t].n[K - 1];
        w.cstart[k][v] = v;
    }
}

// Study switch "no de-duplication" (the first arm of the paper's reuse ablation): lookup l is row slot l and a group of
// its own at every prefix level, so nothing is shared: every lookup rebuilds its whole chain of products.
// Lookups with a row id outside the table keep the row 0 (the pooling pass skips them by their id).
__global__ void __launch_bounds__(256) k_nodedup_levels(WsView w)
{
    tt_pdl_enter();
    const int K = w.K;
    const int64_t L = w.L < (int64_t)w.cap[K] ? w.L : (int64_t)w.cap[K];
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (first == 0) {
        if (w.L > (int64_t)w.cap[K]) atomicOr(w.status, TT_EMB_STATUS_OVERFLOW);
        for (int k = 1; k <= K; ++k) {
            w.counters[CTR_LEVEL0 + k] = (uint32_t)L;
            if (k < K) w.cstart[k][L] = (uint32_t)L;
        }
    }
    if (first <= w.T)
        for (int k = 1; k <= K; ++k) {
            const int64_t v = w.tl_start[first];
            w.tb[k][first] = (uint32_t)(v < L ? v : L);
        }
    int t = 0;
    for (int64_t l = first; l < L; l += (int64_t)gridDim.x * blockDim.x) {
        if (!(w.tl_start[t] <= l && l < w.tl_start[t + 1])) t = tt_find_table64(w.tl_start, w.T, l);
        const TableDesc& td = w.tdesc[t];
        const int64_t g = tt_index(w, l);
        if (g < 0 || g >= td.N) atomicOr(w.status, TT_EMB_STATUS_INDEX);
        uint32_t v = (g >= 0 && g < td.N) ? (uint32_t)g : 0u;
        for (int k = K; k >= 1; --k) {
            w.val[k][l] = v;
            if (k < K) w.cstart[k][l] = (uint32_t)l;
            if (w.parent[k]) w.parent[k][l] = (uint32_t)l;
            v /= (uint32_t)td.n[k - 1];
        }
    }
}

// 0: a kernel per step; 1: one cluster of sixteen SMs (group_cluster.cu) from the prefix levels on; 2: one cluster for everything;
// 3: one cluster for the scans of the prefix levels, all of them at once; links, the digit-major list and the schedule over all SMs.
// The cluster saves a dozen launches and loses where a step has work for more SMs: scans and links of large prefix spaces, marks
// and scan of long row bitmaps, checks of many offsets.  Forward calls with 0 / 1 / 2, us (L2 flushed in between): row bitmap of 31
// k words, one table, 1 k lookups 83 / 58 / 54, 16 k 94 / 69 / 60, 33 k 103 / 73 / 67; 125 k words, one table, 1 k 85 / 60 / 63, 16
// k 96 / 73 / 73; two tables, 94 k words, 16 k 91 / 69 / 69; four, 125 k words, 16 k 91 / 65 / 71; eight, 125 k words, 33 k 102 /
// 73 / 83; eight, 0.5 M words, 8 k 106 / 77 / 110; thirty small tables, 16 k 110 / 77 / 99: with several tables the line of mode 2
// lies lower than it has been drawn. Prefix bitmaps (0 / 1), spread rows unless stated: up to 8 k words whatever the batch: two
// tables of 40 M rows, popular rows first, 33 k lookups 136 / 118, 2 M 458 / 433, 8 M 888 / 888; between 8 k and 16 k words only
// with few lookups, which leave most of the prefixes out: 12 k words, eight tables, 33 k 134 / 112, 2 M 475 / 470, 8 M 850 / 843;
// 16 k words, four tables, 33 k 153 / 138, 2 M 553 / 566, 8 M 962 / 980; past it 20 k words, 33 k 157 / 134, 2 M 571 / 583; 46 k
// words, 33 k 210 / 196, 0.26 M 335 / 333, 2 M 784 / 831. Offsets (20 k lookups, 0 / 1 / 2): 0.2 M 123 / 97 / 101, 1 M 258 / 230 /
// 237.
// Mode 3 against 0, whole calls, us: 17 k words, 3 k lookups 182 / 157, 10 k 202 / 176, 0.3 M 249 / 220 (forward); 20 k words, 0.55 M 616 / 572;
// 27 k words, 30 k 214 / 195 (forward), 4 M 1154 / 1126; 39 k words, 24 M 4305 / 4227; 48 k words, 99 M 5440 / 5383; but 165 k words, 69 M
// 14461 / 14503 (the scans of sixteen SMs).  86 drawn calls past mode 1: 0.954 of their time; one slower by more than 1 % (fifty-five tables,
// bags of one, popular rows first, 502 / 525: units of equal counts).  Four cores, whose units have equal costs: 16 k words, 2 k lookups
// 299 / 277, 31 k words, 0.14 M 518 / 491.
// Mode 3 against 1, units of equal counts: 12 k words, 25 k lookups 199 / 168, 0.9 M 804 / 763, 14 k words, 0.8 M 683 / 624; 4 k to 8 k words,
// 0.1 M to 0.6 M 0.96 to 0.99 of the call; 3.5 k words, 4 M 708.5 / 698.5; but 1.5 k words, 0.5 M 240.6 / 237.5 and 0.7 M 216.2 / 217.7, 1.3 k words, 0.3 M 388 / 391,
// 7 k words, 31 k 229 / 233, 0.2 k words, 12 k 98 / 102, 0.3 M 276 / 279.  Equal costs: 8 k words, four cores, 0.5 M 326 / 331.
// 9 k to 15 k words, 1.1 M to 2 M lookups, 28 calls of seven shapes, rank 8 to 32, popular rows first and spread: 0.93 to 0.98 of the forward
// (155 / 143, 207 / 196, 431 / 403, 376 / 362), 0.97 to 0.99 of the training call (370 / 360, 1129 / 1101, 3620 / 3595).
// All that by words of whole scan tiles; with few words in them (TT_CLUSTER_SPREAD_WORDS, the possible prefixes alone) mode 1 is the shorter: rank 32, mode
// 1 / 3, forward, us: 0.25 k words, 0.16 M lookups 91.3 / 93.3; 0.5 k, 0.16 M 96.4 / 97.4, 97.8 / 96.7, 0.5 M 130 / 127.5; 0.8 k, 70 k 94.6 / 93.1, 0.16 M 107.5 / 105.2; 1.3 k,
// 0.16 M 130 / 125.  (Not past 12 k words of whole tiles, where mode 2 would have the fewer lookups: 32 tables of 2 k rows, 25 k, training 127 / 111.)
#define TT_CLUSTER_SCAN_WORDS (3u << 15)
#define TT_CLUSTER_SPREAD_WORDS 512u
#define TT_CLUSTER_ANY_WORDS (1u << 13)
#define TT_CLUSTER_LEVEL_WORDS (1u << 14)
#define TT_CLUSTER_LEVEL_LOOKUPS (1 << 21)
#define TT_CLUSTER_ROW_WORDS (1u << 17)
#define TT_CLUSTER_LOOKUPS (1 << 15)
#define TT_CLUSTER_OFFSETS (1 << 18)
// whether the presence bitmaps of the prefix levels can be written from the bits of the level below (tt_level_words)
static bool tt_prefix_bits(const tt_emb* h)
{
    for (int t = 0; t < h->T; ++t)
        for (int k = 1; k < h->K; ++k)
            if (h->tab[t].n[k] > TT_BITS_RADIX) return false;
    return true;
}
static int tt_use_cluster(const tt_emb* h)
{
    const WsView& w = h->v;
    if (!h->cluster_ok || w.ablation) return 0;
    uint32_t words = w.K >= 3 ? w.ttotal_words[w.K - 1] : 0u;
    for (int k = 1; k < w.K; ++k)
        if (w.total_words_l[k] > words) words = w.total_words_l[k];
    const bool few_words = words <= (w.L <= TT_CLUSTER_LEVEL_LOOKUPS ? TT_CLUSTER_LEVEL_WORDS : TT_CLUSTER_ANY_WORDS);
    const bool spread = h->warp_groups && w.K >= 3 &&
                        (words >= 12288 ? w.L >= 1 << 14 : words >= 3072 && w.L >= 1 << 15 && w.ttotal_words[w.K - 1] >= TT_CLUSTER_SPREAD_WORDS);
    // (L <= capU: the digit-major list has room for all the prefixes that the row ids mark)
    if ((!few_words || spread) && words <= TT_CLUSTER_SCAN_WORDS && w.K >= 3 && w.L <= h->capU && tt_prefix_bits(h)) return 3;
    if (!few_words) return 0;
    return w.total_words <= TT_CLUSTER_ROW_WORDS && w.L <= TT_CLUSTER_LOOKUPS && (int64_t)w.T * w.B <= TT_CLUSTER_OFFSETS ? 2 : 1;
}

cudaError_t tt_launch_grouping(tt_emb* h, cudaStream_t s)
{
    WsView& w = h->v;
    cudaError_t e;
    const int cluster = tt_use_cluster(h);
    w.equal_units = (cluster != 0 && (h->warp_groups || w.K == 2)) || (w.ablation & 2) ? 1 : 0;   // (units of K = 2 are ranges of rows)
    // Prefix bitmaps from the bits of the level below, before any scan.  With the row scan as kernels of their own, the two longest are written
    // by CTAs beside it: in the cluster, sixteen SMs took 9 us for the 9 k words of 8 tables, all on the way of what follows.  Calls,
    // before / after, us: 8 tables, 8 k lookups 78 / 63, 1.6 M 618 / 602 (training); one table, 0.7 M lookups 231 / 222, four cores 342 / 329;
    // at most one / two / four such CTAs per SM: 65.7 / 63.6 / 62.8 and 604.7 / 602.2 / 601.8.
    const bool bits = tt_prefix_bits(h);
    if (cluster == 2) return tt_launch_group_cluster(h, true, bits ? w.K : 0, true, s);
    unsigned side = 0;           // a warp per word of the largest of the bitmaps that are written beside the row scan
    if ((cluster == 1 && bits) || cluster == 3) {
        uint32_t words = w.total_words_l[w.K - 1];
        if (w.K >= 3 && w.total_words_l[w.K - 2] > words) words = w.total_words_l[w.K - 2];
        side = (words + TT_SCAN_THREADS / 32 - 1) / (TT_SCAN_THREADS / 32);
        if (side > (unsigned)h->sm_count * 4) side = (unsigned)h->sm_count * 4;
    }
    // status word, counters and row bitmap lie side by side (with a memset each: 8 tables, 8 k lookups, call 63.1 us instead of 60.8)
    if ((e = cudaMemsetAsync(w.status, 0, TT_STATUS_BYTES + (w.ablation & 4 ? 0 : (size_t)w.total_words * sizeof(uint2)), s)) != cudaSuccess) return e;
    const int64_t nb = (int64_t)w.T * w.B + 1;
    int g0 = (int)((nb + 255) / 256);
    if (g0 > h->sm_count * 8) g0 = h->sm_count * 8;
    if (w.ablation & 4) {
        if ((e = tt_launch_pdl(k_check_offsets, dim3(g0), dim3(256), 0, s, w)) != cudaSuccess) return e;
        tt_note_launch();
        if ((e = tt_launch_pdl(k_nodedup_levels, dim3(h->sm_count * 8), dim3(256), 0, s, w)) != cudaSuccess) return e;
        tt_note_launch();
        return cudaGetLastError();
    }
    if (cluster == 0 && tt_digit_major(w) && (e = cudaMemsetAsync(w.tbm[w.K - 1], 0, (size_t)w.ttotal_words[w.K - 1] * sizeof(uint2), s)) != cudaSuccess) return e;
    {
        int64_t want = (w.L + 1023) / 1024;
        const bool fused = w.L <= TT_FUSED_INGEST;
        if (fused && want < g0) want = g0;
        if (want > h->sm_count * 8) want = h->sm_count * 8;
        if (!fused) {
            if ((e = tt_launch_pdl(k_check_offsets, dim3(g0), dim3(256), 0, s, w)) != cudaSuccess) return e;
            tt_note_launch();
        }
        if ((e = tt_launch_pdl(fused ? k_mark<true> : k_mark<false>, dim3((unsigned)want), dim3(256), 0, s, w, side && tt_digit_major(w) ? 1 : 0)) != cudaSuccess) return e;
        tt_note_launch();
    }
    // short bitmaps in finer tiles, so that they spread over the SMs
    const unsigned ptiles = (unsigned)(TT_HEAD_TILES * w.T) + w.rest_tiles;
    if (w.total_words <= TT_PSCAN_FINE_WORDS && w.L >= TT_PSCAN_FINE_LOOKUPS && w.L >= (int64_t)w.total_words) {
        PopScan<TT_SCAN_THREADS * 2> ps{w, side};
        e = tt_scan<decltype(ps), 2>(ps, w.total_words, w.scan_tmp, s, ptiles * (TT_SCAN_ITEMS / 2), side);
    } else if (w.total_words <= TT_PSCAN_WORDS) {
        PopScan<TT_SCAN_THREADS * TT_PSCAN_ITEMS> ps{w, side};
        e = tt_scan<decltype(ps), TT_PSCAN_ITEMS>(ps, w.total_words, w.scan_tmp, s, ptiles * (TT_SCAN_ITEMS / TT_PSCAN_ITEMS), side);
    } else {
        PopScan<TT_SCAN_TILE> ps{w, side};
        e = tt_scan(ps, w.total_words, w.scan_tmp, s, ptiles, side);
    }
    if (e != cudaSuccess) return e;
    if (cluster == 1) return tt_launch_group_cluster(h, false, side ? (w.K >= 4 ? w.K - 2 : 1) : 0, true, s);
    if (cluster == 3) {
        if ((e = tt_launch_group_cluster(h, false, w.K >= 4 ? w.K - 2 : 1, false, s)) != cudaSuccess) return e;
        if ((e = tt_launch_pdl(k_links, dim3(h->sm_count * 8, w.K - 1), dim3(256), 0, s, w, 0, w.equal_units)) != cudaSuccess) return e;
        tt_note_launch();
        return cudaGetLastError();
    }
    for (int k = w.K - 1; k >= 1; --k) {
        {
            const uint32_t want = (w.total_words_l[k] + 7u) / 8u;   // a warp per word
            const uint32_t g = want < (uint32_t)h->sm_count * 8u ? (want ? want : 1u) : (uint32_t)h->sm_count * 8u;
            if ((e = tt_launch_pdl(k_prefix_bits, dim3(g), dim3(256), 0, s, w, k)) != cudaSuccess) return e;
            tt_note_launch();
        }
        LevelScan<> ls{w, k};
        if ((e = tt_scan<LevelScan<>, TT_LSCAN_ITEMS>(ls, w.total_words_l[k], w.scan_tmp, s)) != cudaSuccess) return e;
        if ((w.ablation & 1) && k == w.K - 1) {   // the scan still sets the bits of level K-2; its nodes are replaced
            if ((e = tt_launch_pdl(k_unique_groups, dim3(h->sm_count * 8), dim3(256), 0, s, w)) != cudaSuccess) return e;
            tt_note_launch();
        }
    }
    // after all the scans: a node's links look into the levels on both sides
    if ((e = tt_launch_pdl(k_links, dim3(h->sm_count * 8, w.K - 1), dim3(256), 0, s, w, tt_digit_major(w) ? 1 : 0, 0)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- digit-major lists, schedule

__global__ void __launch_bounds__(256) k_tmark(WsView w, int k)
{
    tt_pdl_enter();
    const uint32_t count = w.counters[CTR_LEVEL0 + k];
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < count; v += gridDim.x * blockDim.x)
        tt_tmark_node(w, w.tdesc[tt_find_table(w.tb[k], w.T, v)], k, v);
}

__global__ void __launch_bounds__(256) k_tfill(WsView w, int k, int costs)
{
    tt_pdl_enter();
    const uint32_t count = w.counters[CTR_LEVEL0 + k];
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < count; v += gridDim.x * blockDim.x)
        tt_tfill_node(w, w.tdesc[tt_find_table(w.tb[k], w.T, v)], k, v, costs != 0);
}

static cudaError_t launch_tfill(tt_emb* h, int k, bool costs, bool scan, cudaStream_t s)
{
    WsView& w = h->v;
    cudaError_t e;
    TPopScan<> tp{w, k};
    if (scan && (e = tt_scan(tp, w.ttotal_words[k], w.scan_tmp, s)) != cudaSuccess) return e;
    if ((e = tt_launch_pdl(k_tfill, dim3(h->sm_count * 8), dim3(256), 0, s, w, k, costs ? 1 : 0)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

cudaError_t tt_launch_tlist(tt_emb* h, int k, cudaStream_t s)
{
    WsView& w = h->v;
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.tbm[k], 0, (size_t)w.ttotal_words[k] * sizeof(uint2), s)) != cudaSuccess) return e;
    if ((e = tt_launch_pdl(k_tmark, dim3(h->sm_count * 8), dim3(256), 0, s, w, k)) != cudaSuccess) return e;
    tt_note_launch();
    return launch_tfill(h, k, false, true, s);
}

// natural sweep order (study switch "no prefix reuse")
__global__ void __launch_bounds__(256) k_costs(WsView w)
{
    tt_pdl_enter();
    const uint32_t count = w.counters[CTR_LEVEL0 + w.K - 1];
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < count; g += gridDim.x * blockDim.x)
        w.cost[g] = tt_group_cost(w, w.tdesc[tt_find_table(w.tb[w.K - 1], w.T, g)], g);
}

// Partition of the sweeps and of the pooling pass, once per forward: the group range of every work unit (the sweeps of the
// forward and of the backward read two words instead of bisecting the cost array at the start of every CTA, two chains of
// ~20 dependent loads each: contraction 2.27 -> 2.16 ms, backward sweeps 4.49 -> 4.43 ms on the 60-table training step) and
// the first bag of every share, where there are many bags per share or the offsets are flagged (otherwise the offsets check has written
// it).  One thread each, so that the bisections run side by side.
__global__ void __launch_bounds__(128) k_partition(WsView w)
{
    tt_pdl_enter();
    const int64_t units = (int64_t)w.T * w.units_per_table;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = first; u < units; u += step) tt_unit_bounds(w, (int)u);
    if (tt_pool_bounds_missing(w))
        for (int64_t ci = first; ci <= w.pool_shares; ci += step) tt_pool_bound(w, ci);
}

cudaError_t tt_launch_schedule(tt_emb* h, cudaStream_t s)
{
    WsView& w = h->v;
    cudaError_t e;
    const int cluster = tt_use_cluster(h);
    if (cluster == 1 || cluster == 2) return cudaSuccess;   // done with the grouping
    if (cluster == 0 || !w.equal_units) {
        if (tt_digit_major(w)) {
            if ((e = launch_tfill(h, w.K - 1, true, cluster == 0, s)) != cudaSuccess) return e;
        } else if (w.K >= 3) {
            if ((e = tt_launch_pdl(k_costs, dim3(h->sm_count * 8), dim3(256), 0, s, w)) != cudaSuccess) return e;
            tt_note_launch();
        }
        if (w.K >= 3) {
            CostScan<> cs{w};
            if ((e = tt_scan<CostScan<>, TT_CSCAN_ITEMS>(cs, w.cap[w.K - 1], w.scan_tmp, s)) != cudaSuccess) return e;
        }
    }
    int64_t want = (int64_t)w.T * w.units_per_table;
    if (want < w.pool_shares + 1) want = w.pool_shares + 1;
    want = (want + 127) / 128;
    if (want > h->sm_count * 16) want = h->sm_count * 16;
    if ((e = tt_launch_pdl(k_partition, dim3((unsigned)want), dim3(128), 0, s, w)) != cudaSuccess) return e;
    tt_note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- export (inspection)

// first leaf (level-K node) under node v of level k
__device__ __forceinline__ uint32_t tt_first_leaf(const WsView& w, int k, uint32_t v)
{
    for (int j = k; j < w.K; ++j) v = w.cstart[j][v];
    return v;
}

__global__ void k_export_mult(WsView w, int table)
{
    // lookups per distinct row of one table -> cursor[] (scratch), via the rank structure
    const TableDesc& td = w.tdesc[table];
    const int64_t lo = w.tl_start[table], hi = w.tl_start[table + 1];
    for (int64_t l = lo + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < hi; l += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = tt_index(w, l);
        if (g < 0 || g >= td.N) continue;
        const uint2 e = w.bm[td.word_base + ((uint32_t)g >> 5)];
        const uint32_t slot = e.y + __popc(e.x & ((1u << (g & 31)) - 1u));
        if (slot < w.cap[w.K]) atomicAdd(&w.cursor[slot], 1u);
    }
}

__global__ void k_export_level(WsView w, int table, int k, int64_t* vals, int32_t* rc, int32_t* lc, int have_mult)
{
    const uint32_t v0 = w.tb[k][table], v1 = w.tb[k][table + 1];
    for (uint32_t v = v0 + blockIdx.x * blockDim.x + threadIdx.x; v < v1; v += gridDim.x * blockDim.x) {
        if (vals) vals[v - v0] = (int64_t)w.val[k][v];
        const uint32_t l0 = tt_first_leaf(w, k, v);
        const uint32_t l1 = (v + 1 < w.counters[CTR_LEVEL0 + k]) ? tt_first_leaf(w, k, v + 1) : w.counters[CTR_LEVEL0 + w.K];
        if (rc) rc[v - v0] = (int32_t)(l1 - l0);
        if (lc && have_mult) {
            uint32_t s = 0;
            for (uint32_t u = l0; u < l1; ++u) s += w.cursor[u];
            lc[v - v0] = (int32_t)s;
        }
    }
}

cudaError_t tt_launch_export_level(tt_emb* h, int table, int level, int64_t* vals, int32_t* rc, int32_t* lc, cudaStream_t s)
{
    WsView& w = h->v;
    if (lc) {
        cudaError_t e = cudaMemsetAsync(w.cursor, 0, (size_t)w.cap[w.K] * sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
        k_export_mult<<<h->sm_count * 4, 256, 0, s>>>(w, table);
        tt_note_launch();
    }
    k_export_level<<<h->sm_count * 4, 256, 0, s>>>(w, table, level, vals, rc, lc, lc ? 1 : 0);
    tt_note_launch();
    return cudaGetLastError();
}

__global__ void k_export_inverse(WsView w, int table, int32_t* inv)
{
    const TableDesc& td = w.tdesc[table];
    const int64_t lo = w.tl_start[table], hi = w.tl_start[table + 1];
    const uint32_t base = w.tb[w.K][table];
    for (int64_t l = lo + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < hi; l += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = tt_index(w, l);
        int32_t r = -1;
        if (g >= 0 && g < td.N) {
            const uint2 e = w.bm[td.word_base + ((uint32_t)g >> 5)];
            r = (w.ablation & 4) ? (int32_t)(l - lo) : (int32_t)(e.y + __popc(e.x & ((1u << (g & 31)) - 1u)) - base);
        }
        inv[l - lo] = r;
    }
}

cudaError_t tt_launch_export_inverse(tt_emb* h, int table, int32_t* inv, cudaStream_t s)
{
    k_export_inverse<<<h->sm_count * 4, 256, 0, s>>>(h->v, table, inv);
    tt_note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------- core layout conversion

__global__ void k_pack(const float* __restrict__ src, float* __restrict__ dst, int rp, int n, int d, int rn, int to_canonical)
{
    // canonical [n][rp][d][rn]  <->  index order [rp][n][d][rn]
    const int64_t total = (int64_t)rp * n * d * rn;
    const int inner = d * rn;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(c % inner);
        const int64_t q = c / inner;
        const int a = (int)(q % rp);
        const int i = (int)(q / rp);
        const int64_t o = ((int64_t)a * n + i) * inner + x;
        if (to_canonical) dst[c] = src[o]; else dst[o] = src[c];
    }
}

cudaError_t tt_launch_pack(const TableDesc& td, int core, const float* src, float* dst, bool to_canonical, cudaStream_t s)
{
    const int64_t total = td.core_floats[core];
    int grid = (int)((total + 255) / 256);
    if (grid > 4096) grid = 4096;
    if (grid < 1) grid = 1;
    k_pack<<<grid, 256, 0, s>>>(src, dst, td.r[core], td.n[core], td.d[core], td.r[core + 1], to_canonical ? 1 : 0);
    tt_note_launch();
    return cudaGetLastError();
}
