// Internal declarations shared by the translation units of libtt_emb.so (sm_100a only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "tt_emb.h"

#define TT_MAXK 4
#define TT_SCAN_THREADS 256
#define TT_SCAN_ITEMS 16
#define TT_SCAN_TILE (TT_SCAN_THREADS * TT_SCAN_ITEMS)  // elements per scan tile
#define TT_POOL_MAX_SHARES 131072                       // shares of the lookups that the pooling warps take in order
#define TT_HEAD_TILES 4                                 // leading scan tiles of a table that are emitted first (see PopScan)
#define TT_LSCAN_ITEMS 2                                // the short scans of the prefix-level bitmaps
#define TT_LSCAN_TILE (TT_SCAN_THREADS * TT_LSCAN_ITEMS)
#define TT_CSCAN_ITEMS 4                                // the scan of the group costs
#define TT_PSCAN_ITEMS 4                                // the scan of row bitmaps of up to TT_PSCAN_WORDS words
#define TT_PSCAN_WORDS (1u << 21)
// up to so many words, from so many lookups and from one per word on, tiles of half that size: the densest tile, whose rows one CTA
// lists, takes half as long, and there are twice as many others.  Forward calls of 1, 2, 4 and 8 tables of 1 M to 40 M rows, D = 16, with
// 512-word tiles relative to 1024: up to 0.5 M words, 0.26 to 4 M lookups, popular rows first 0.95 to 0.99 (one table of 31 k words, 1 M
// lookups 144.4 / 138.4 us; 0.5 M words, 0.26 M lookups 111.6 / 105.5), spread rows 0.96 to 1.0; 16 k and 65 k lookups 0.97 to 1.03; 0.78 M
// words 0.98 to 1.02 (spread 173 / 175); 1 M words and more 0.99 to 1.04, with 16 k to 65 k lookups 1.02 to 1.08 (81 / 85).  The line
// lies between 0.5 and 0.78 M words.
#define TT_PSCAN_FINE_WORDS 655360u
#define TT_PSCAN_FINE_LOOKUPS (1 << 18)
// most lookups whose marking pass also checks the offsets: one launch less, but the tables' ranges come from all over the
// offsets (99 M lookups, 60 tables: grouping 0.76 ms with two kernels, 0.81 ms with one; 0.5 M, 8 tables: 3 us shorter)
#define TT_FUSED_INGEST (1 << 22)
// fewest groups of a work unit; 4x as many for D = 128, rank 32, whose warps each reuse a 32 KB slice over their groups.
// Sweeps with at least 4 / 8 / 16 / 32 / 64 groups per unit, forward + backward, us: 8 tables x 8 k groups (rank 16) 385 / 352 /
// 325 / 319 / 343; 4 tables x 9 k (D = 32, rank 8) 119 / 117 / 107 / 122 / 188; four cores, 4.7 k groups 178 / 173 / 170 / 235;
// D = 128, rank 32, 27 k groups (forward) 236 / 164 / 145 / 137 / 129.
// D = 32 and 16 with ranks 16 and 32 take eight groups per warp in both sweeps, 32 per round of a CTA's four warps.  Where the
// groups fill the chip twice over with units of 16 (TT_PAIRED_GROUPS per SM: six such CTAs fit an SM), they get units of at
// most 32, so that every warp has its eight (training call of 8 tables, 8 M lookups of spread rows, 180 k groups, rank 32, units
// of 16 / 32: 1973 / 1700 us; 15 % to 18 % on 0.1 M to 8 M lookups); below, finer units balance better than full warps (33
// tables, 12 k groups 247 / 275; 18 tables, 69 bags each 1.12 times longer with 32).  At least 32 instead of at most 32 leaves
// units of 33 groups, whose fifth batch costs a second round (53 tables, 19 k groups, forward 282 / 334).
#define TT_UNIT_GROUPS 16
#define TT_PAIRED_GROUPS (2 * 6 * TT_UNIT_GROUPS)
// ... and of the any-shape sweeps, whose CTAs take a batch of groups at a time (3x3x5, 29 k groups, forward + backward sweep
// with at least 1 / 4 / 8 / 16 groups: 332 / 285 / 252 / 253 us; 8x8 with K = 2, 420 k lookups, whole call 1.16 ms with 8, 1.68 with 16)
#define TT_UNIT_GROUPS_ANY 8
// ... and with last dim factors that are no multiples of four, whose backward takes rows to a thread, at least TT_UNIT_ROWS_ODD rows too, up
// to 32 groups, where there are groups enough.  3x3x5, backward sweep, us, units of 4 / 8 / 16 / 32 groups: 1.8 rows a group, 26 k groups 76 /
// 56 / 48 / 57; 1.4 rows, 17 k groups 59 / 35 / 31 / 32; 8 rows, 29 k groups 104 / 97 / 106 / 133; with at least 24 / 32 / 48 rows the first
// 46 / 40 / 42 (forward sweep, with 8 groups and with 32 rows: 40 / 33).
#define TT_UNIT_ROWS_ODD 32
// Batches of few groups: below TT_FEW_LIMIT groups per CTA of TT_FEW_UNITS on every SM, the sweeps cut the tables' groups into that many
// equal parts of at least TT_FEW_GROUPS, and each of a CTA's warps takes a quarter.  A warp that takes its four or eight at once fetches
// one slice after the other, 3 us each for 4 KB, 12 us for 32 KB, while most of the chip idles.  Forward / backward sweep, us, in the
// schedule's units and so cut: D = 128, rank 32, 1.0 k groups 180 / 96 and 23 / 19; D = 32, rank 32, 0.8 k 52 / 59 and 19 / 23; rank 16,
// 1.2 k 28 / 43 and 17 / 23; four cores, 0.5 k 56 / 70 and 29 / 37.  Limits of 4 / 8 / 12: 150 drawn calls 0.965 / 0.961 / 0.959 of
// their time (geometric mean), but above 8 cheap and dear groups in equal parts cost some 3 %.  Six CTAs per SM: as four.
// The kernels that can do this have more CTAs than there are units, so theirs go table by table first: the CTAs without work are the last.
// (Unit by unit first, as the others', a table's idle CTAs held up the next one's: 4 tables, D = 128, rank 32, 9 k groups, forward sweep 123
// us, 98 now, 88 without the extra CTAs; D = 16 and 64, rank 32, 5 k groups 36 and 43 / 29 and 35 / 29 and 35.)  They are launched where at most
// TT_FEW_MAYBE times as many groups are possible by the lookups and the tables: 8 times, 4 tables, D = 128, rank 32, 30 k possible, 0.14 M lookups,
// training call 616 without, 638 with them; no drawn call with that many possible had few.
#define TT_FEW_UNITS 4
#define TT_FEW_GROUPS 4
#define TT_FEW_LIMIT 8
#define TT_FEW_MAYBE 4
#define TT_STATUS_BYTES 512   // status word and counters (16 + 64 words) with their guard bytes, up to the row bitmap behind them
#define TT_GUARD 0xA5         // guard bytes behind the other workspace regions
#define TT_UNIT_ROWS 64   // fewest rows of a unit of a K = 2 table
#define TT_DE_CHUNK 1024                                  // sorted lookups per warp in the dE segment reduction, at most (up to 134 M lookups)
#define TT_NUM_STAGES 33                                // 0..8 pipeline stages, 9..20 forward sweep variants -1..10, 21..32 backward sweep variants
#define TT_STRIPES 8                                     // L2-resident partial copies of the last core's gradient
#define TT_NUM_MIDFAST 11                                // tensor-core instances of the middle-core backward (backward.cu)
#define TT_NUM_VARIANTS 11                               // register-tiled shape variants (forward.cu)

// Per-table descriptor, resident in the workspace.  k below is 0-based (core k+1 of the paper).
struct TableDesc {
    int64_t N;
    int32_t n[TT_MAXK];
    int32_t d[TT_MAXK];
    int32_t r[TT_MAXK + 1];
    int32_t P[TT_MAXK + 1];             // P[0] = 1, P[k] = d_1 * .. * d_k
    int32_t slice_floats[TT_MAXK];      // r[k] * d[k] * r[k+1]
    int64_t core_floats[TT_MAXK];       // n[k] * slice_floats[k]
    float* core[TT_MAXK];
    float* grad[TT_MAXK];
    uint32_t word_base;                 // first 32-row word of this table in the presence bitmap
    uint32_t num_words;
    uint32_t rest_base;                 // scan tiles of the tables before this one, their first TT_HEAD_TILES each left out
    uint32_t lword_base[TT_MAXK];       // the same for the presence bitmaps of the length-k prefixes, k = 1..K-1
    uint32_t suffix[TT_MAXK];           // n_{k+1} * .. * n_K: row id / suffix[k] = length-k prefix value, k = 1..K-1
    uint32_t tword_base[TT_MAXK];       // same for the digit-major ("transposed") node bitmaps, levels 2..K-1
    uint32_t tnum_words[TT_MAXK];
    uint32_t prefix_space[TT_MAXK + 1]; // n_1 * .. * n_k (number of possible length-k prefixes), k = 1..K-1
    int64_t gpart_off;                  // float offset of this table's last core inside one stripe
    int32_t units;                      // work units (CTAs) this table is cut into
    int32_t unit_base;                  // first global unit id
    int32_t sgd_mask;                   // bit k: the fused backward + SGD call updates core k inside the kernel that finalises its gradient
    int32_t unit_groups;                // a work unit holds at least this many groups
    int32_t fast;                       // register-tiled kernel variant for this table's shapes, -1 = generic path
    int32_t midfast[TT_MAXK];           // same for the middle-core backward of level k (index k), -1 = generic
};

// Device-side view of the workspace handed to kernels by value.
struct WsView {
    int32_t T, K, D;
    int32_t ablation;                   // study switches: bit 0 no prefix reuse, bit 1 static (equal-count) schedule,
                                        // bit 2 no de-duplication (every lookup is its own row and its own group; implies bit 0)
    int32_t equal_units;                // 1: work units of equal group counts instead of equal costs (study switch; schedules made in
                                        // one cluster for tables swept by warps, without the scan of the costs: group_cluster.cu)
    int32_t cost_shift;                 // cost unit of the schedule = 2^cost_shift FMAs
    uint32_t paired_groups;             // from this many groups on, units of shapes with eight groups per warp hold 2 * TT_UNIT_GROUPS
    uint32_t few_units;                 // sweep CTAs that run at once: few groups are cut into about that many units (tt_sweep_unit)
    float few_share, cta_share;         // 1 / few_units, 1 / CTAs of a table in the sweeps
    float fused_lr;                     // != 0: the kernels that finalise a gradient also apply G -= fused_lr * dG (cores in sgd_mask)
    int32_t stride[TT_MAXK + 1];        // floats per node of the level-k partial-product buffers (max over tables)
    int64_t B, L;                       // current batch / lookups
    int64_t capU;                       // capacity in distinct rows
    uint32_t cap[TT_MAXK + 1];          // node capacity per level 1..K
    uint32_t total_words;
    uint32_t ttotal_words[TT_MAXK];
    int32_t* status;
    uint32_t* counters;                 // [k] = number of level-k nodes (k = 1..K); [8+k] transposed counts
    TableDesc* tdesc;
    int32_t* vlist;                     // [0,T): table ids grouped by kernel variant (generic first); [T,2T): all tables;
                                        // largest tables first inside each list
    int64_t* tl_start;                  // [T+1] first lookup of each table
    uint2* bm;                          // {32 presence bits, number of set bits before this word (global)}
    uint2* bml[TT_MAXK];                // the same for the length-k prefixes, k = 1..K-1 (one bit per possible prefix)
    uint32_t total_words_l[TT_MAXK];
    uint32_t rest_tiles;                // scan tiles of the row bitmap beyond the first TT_HEAD_TILES of every table
    uint32_t* scan_tmp;
    uint32_t* val[TT_MAXK + 1];         // level k: prefix value within the table (k = K: row id)
    uint32_t* cstart[TT_MAXK + 1];      // level k < K: first child (level k+1 node); [count] = sentinel
    uint32_t* parent[TT_MAXK + 1];      // levels 3..K-1: parent node at level k-1 (null elsewhere: nothing reads it)
    uint32_t* tb[TT_MAXK + 1];          // [T+1] node range of each table at level k
    uint32_t* cost;                     // [cap_{K-1}+1] exclusive scan of per-group cost (+ total)
    int64_t pool_shares;                // shares of the lookups in the pooling pass (0: it takes no shares)
    int64_t* pool_bounds;               // [shares + 1] first bag of every share of the pooling pass (group.cuh)
    uint2* unit_rng;                    // [T * units per table] group range of every work unit (tt_unit_bounds)
    int32_t units_per_table;
    float* pbuf[TT_MAXK + 1];           // partial products P_k of level-k nodes, 2 <= k <= K-2
    float* E;                           // [capU][D] rows (forward) / dE (backward)
    // backward
    uint32_t* cnt;                      // [capU+1] lookups per distinct row -> segment starts inside their tiles (tt_seg_start)
    uint32_t* cursor;                   // [capU]
    uint2* pairs;                       // [L] bags sorted by slot (uint32, behind them the pairs' ranks), or (bag, factor) with weights or mean pooling
    uint32_t* chunk_slot;               // slot of the first sorted position of every dE chunk (in the space of pool_bounds)
    uint32_t* chunk_ctr;                // pieces of the segments that cross chunk borders, counted as they arrive (behind them)
    uint2* upairs;                      // [L] (slot, bag) in lookup order, written by the pooling kernel (null: forward only)
    float* dP[TT_MAXK + 1];             // dP_k per level-k node, 2 <= k <= K-1
    float* Y[TT_MAXK + 1];              // per level-k node: its contribution to dP_{k-1} of its parent
    float* carry;                       // [chunks][2][D] pieces of the segments that cross a chunk border
    uint32_t de_chunk_log;              // 1 << de_chunk_log sorted lookups per warp in the dE segment reduction
    float* gpart;                       // [TT_STRIPES][gpart_stride] partial copies of all tables' last-core gradients
    int64_t gpart_stride;               // floats per stripe
    uint2* tbm[TT_MAXK + 1];            // digit-major node bitmaps, levels 2..K-1
    uint32_t* tnode[TT_MAXK + 1];       // nodes of level k ordered by (table, i_k, parent prefix)
    const int64_t* indices;
    const int64_t* offsets;
    // pooling beyond the plain sum (tt_emb_set_pooling)
    const float* psw;                   // per-lookup weights [L] or null
    float* wsorted;                     // [L] the pairs' ranks where these have factors (weight, or 1 / bag length), backward only
    int32_t pool_mean;                  // 1: mean pooling
    int32_t idx32;                      // 1: `indices` points at int32 row ids (tt_emb_forward_i32)
};

// row id of lookup l (int64 or int32 storage); STREAM: read-once hint
template <bool STREAM = false>
__device__ __forceinline__ int64_t tt_index(const WsView& w, int64_t l)
{
    if (w.idx32) {
        const int32_t* p = reinterpret_cast<const int32_t*>(w.indices) + l;
        return (int64_t)(STREAM ? __ldcs(p) : __ldg(p));
    }
    return STREAM ? __ldcs(w.indices + l) : __ldg(w.indices + l);
}

// whether the pairs of the backward have factors
__host__ __device__ __forceinline__ bool tt_weighted(const WsView& w) { return w.wsorted && (w.psw || w.pool_mean); }

enum { CTR_LEVEL0 = 0 /* +k */, CTR_TLEVEL0 = 8 /* +k */, CTR_COST_TOTAL = 16, CTR_SCAN_TICKET = 32 /* tiles of the running scan that have reported */,
       CTR_POOL_NEXT = 34 /* next share of the lookups to be pooled (shares are handed out in order) */,
       CTR_DIRECT = 40 /* k_direct: CTAs that have reported, their status bits; 1 where the last forward made no grouping, its batch, lookups,
                          idx32; next bag, long bags (direct.cu): twelve words */ };

struct tt_emb {
    int T, K, D;
    int64_t max_batch, max_lookups, capU;
    int enable_backward;
    int enable_weighted;
    int ablation;
    int sm_count;
    int units_total;
    int units_per_table;
    int sweep_ctas;       // CTAs of a table in the sweeps: its units, or more where few groups are cut finer
    int vcount[TT_NUM_VARIANTS + 1];   // tables per variant, index 0 = generic (-1)
    int vbase[TT_NUM_VARIANTS + 1];    // first entry of each variant in vlist
    // middle-core kernels of level k: tables grouped by their variant (index 0 = generic), largest first, in
    // vlist[(2 + k) * T ..); first entry, count and largest n_k of each group
    int mbase[TT_MAXK + 1][TT_NUM_MIDFAST + 1], mcount[TT_MAXK + 1][TT_NUM_MIDFAST + 1], mmaxn[TT_MAXK + 1][TT_NUM_MIDFAST + 1];
    int32_t* vlist_host;
    size_t off_vlist;
    TableDesc* tab;       // host copy [T]
    size_t ws_bytes;
    size_t off_status, off_counters, off_tdesc, off_tlstart, off_bm, off_scan, off_cost, off_E;
    size_t off_bml[TT_MAXK];
    size_t off_val[TT_MAXK + 1], off_cstart[TT_MAXK + 1], off_parent[TT_MAXK + 1], off_tb[TT_MAXK + 1];
    size_t off_pbuf[TT_MAXK + 1], off_dP[TT_MAXK + 1], off_tbm[TT_MAXK + 1], off_tnode[TT_MAXK + 1];
    size_t off_Y[TT_MAXK + 1];
    size_t off_cnt, off_cursor, off_pairs, off_carry, off_gpart, off_wsorted, off_unit_rng, off_pool_bounds;
    // guard bytes after every workspace region (tt_emb_check_guards): [guard_off[i], guard_off[i] + guard_len[i])
    int num_regions;
    size_t guard_off[96], guard_len[96];
    unsigned char guard_value[96];
    const char* region_name[96];
    size_t off_guard_list;      // device copy of the (offset, length) pairs + the check's result word
    void* ws_base;
    bool warp_groups;     // every table is swept by warps that take groups one batch at a time (not by whole CTAs)
    int cluster_ok;       // the device takes the cluster of group_cluster.cu
    int direct_ctas[2];   // resident CTAs per SM of k_direct without / with weights, 0: not asked since the bind
    int pool_grid;        // CTAs of the pooling kernel (tt_plan_pooling)
    float* carry;         // workspace region of v.carry for chunks of TT_DE_CHUNK lookups
    size_t scan_tmp_elems;
    int64_t gpart_floats;
    WsView v;             // filled at bind
    bool bound, have_forward;
    bool timing;
    bool serial;          // timing mode 2: shape-variant kernels run one after the other (per-kernel durations)
    cudaEvent_t ev[TT_NUM_STAGES][2];
    bool ev_valid[TT_NUM_STAGES];
    bool ev_created;
    // side streams for kernels of different shape variants that may overlap (created on first use; the first at bind for training with
    // four cores)
    cudaStream_t side[4];
    cudaEvent_t side_ev[4], fork_ev;
    int side_made;
};

// every kernel launch of the library is noted here (api.cu); read with tt_emb_launch_count
void tt_note_launch(int n = 1);
// remember a failing CUDA call for tt_emb_last_cuda_error (api.cu)
void tt_set_last_cuda_error(cudaError_t e);
// compute capability 10.x device current? (api.cu)
int tt_device_ok(int* sm_count);

// tt_emb_bind; make_streams: with the streams that every backward takes (api.cu)
int tt_bind(tt_emb* h, float* const* core_ptrs, void* workspace, size_t workspace_bytes, cudaStream_t s, bool make_streams);

// fork/join helpers (api.cu): side streams wait for everything enqueued on `s` so far / `s` waits for the side streams
cudaError_t tt_fork(tt_emb* h, cudaStream_t s, int n);
cudaError_t tt_join(tt_emb* h, cudaStream_t s, int n);

// stage timing (api.cu): no-ops unless timing is enabled
cudaError_t tt_stage_begin(tt_emb* h, int stage, cudaStream_t s);
cudaError_t tt_stage_end(tt_emb* h, int stage, cudaStream_t s);

// ---- launchers implemented in the .cu files (all enqueue on `s`, return cudaGetLastError()) ----
cudaError_t tt_launch_grouping(tt_emb* h, cudaStream_t s);
cudaError_t tt_launch_group_cluster(tt_emb* h, bool rows, int level, bool links, cudaStream_t s);
int tt_group_cluster_ok();
cudaError_t tt_launch_schedule(tt_emb* h, cudaStream_t s);
// whether the call may have so few groups that its sweeps cut them finer than the schedule's units (tt_sweep_unit)
inline bool tt_few_groups(const tt_emb* h)
{
    const int64_t most = h->v.L < (int64_t)h->v.cap[h->K - 1] ? h->v.L : (int64_t)h->v.cap[h->K - 1];
    return most <= (int64_t)h->v.few_units * TT_FEW_LIMIT * TT_FEW_MAYBE;
}
cudaError_t tt_launch_tlist(tt_emb* h, int k, cudaStream_t s);   // digit-major list of the level-k nodes (backward, k < K-1)
cudaError_t tt_plan_pooling(tt_emb* h, const float* out);          // grid and shares of the pooling pass, before the schedule
cudaError_t tt_launch_contraction(tt_emb* h, cudaStream_t s);
cudaError_t tt_launch_pooling(tt_emb* h, float* out, cudaStream_t s);
cudaError_t tt_launch_direct(tt_emb* h, float* out, bool* launched, cudaStream_t s);   // the forward without the grouping, where that is shorter
cudaError_t tt_regroup(tt_emb* h, cudaStream_t s);                 // the grouping of such a forward, for the inspection calls
cudaError_t tt_launch_bwd_sort(tt_emb* h, cudaStream_t s);
cudaError_t tt_launch_bwd_dE(tt_emb* h, const float* grad_out, cudaStream_t s);
cudaError_t tt_launch_bwd_contraction(tt_emb* h, cudaStream_t s);
cudaError_t tt_launch_bwd_middle(tt_emb* h, cudaStream_t s);
cudaError_t tt_launch_sgd(tt_emb* h, float lr, bool only_unfused, cudaStream_t s);
cudaError_t tt_launch_export_level(tt_emb* h, int table, int level, int64_t* vals, int32_t* rc, int32_t* lc, cudaStream_t s);
cudaError_t tt_launch_export_inverse(tt_emb* h, int table, int32_t* inv, cudaStream_t s);
cudaError_t tt_launch_pack(const TableDesc& td, int core, const float* src, float* dst, bool to_canonical, cudaStream_t s);

// ---- programmatic dependent launch: the kernels of the forward chain are launched with the attribute below and
// begin with tt_pdl_enter().  A kernel's CTAs may then become resident while its predecessor in the stream is still
// running and wait (griddepcontrol.wait) until that grid has completed and its writes are visible, so the launch
// latency of a chain of short kernels overlaps the previous kernel instead of following it.  Without the attribute
// (or after a non-kernel operation in the stream) the wait returns at once.
__device__ __forceinline__ void tt_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void tt_pdl_enter()
{
    tt_pdl_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... KArgs, class... Args>
static inline cudaError_t tt_launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// a += v as two packed fp32 additions (add.rn.f32x2 of sm_100: two IEEE additions per instruction and lane, the same
// results as four scalar additions; the row sums of the gathers are bound by issue slots)
__device__ __forceinline__ void tt_add4(float4& a, const float4& v)
{
    const float2 lo = __fadd2_rn(make_float2(a.x, a.y), make_float2(v.x, v.y));
    const float2 hi = __fadd2_rn(make_float2(a.z, a.w), make_float2(v.z, v.w));
    a = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// ---- small device helpers ----
__device__ __forceinline__ int tt_find_table(const uint32_t* __restrict__ tb, int T, uint32_t v)
{
    // largest t with tb[t] <= v  (tb non-decreasing, tb[0] = 0)
    int lo = 0, hi = T;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (tb[mid] <= v) lo = mid; else hi = mid;
    }
    return lo;
}

// the same, starting from a table known not to lie after v's (elements of a tile are ascending: the table of the
// tile's first element); usually no step at all
__device__ __forceinline__ int tt_find_table_from(const uint32_t* __restrict__ tb, int T, uint32_t v, int t)
{
    while (t + 1 < T && tb[t + 1] <= v) ++t;
    return t;
}

// out[m*cols + c] = sum_a Pl[m*ra + a] * Bsl[a*cols + c]   (Pl in shared memory, Bsl in global, out anywhere)
__device__ __forceinline__ void tt_mid_product(const float* __restrict__ Pl, const float* __restrict__ Bsl, float* out,
                                               int M, int ra, int cols)
{
    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
        for (int m0 = 0; m0 < M; m0 += 8) {
            float acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = 0.f;
            const int mm = min(8, M - m0);
            for (int a = 0; a < ra; ++a) {
                const float b = __ldg(Bsl + (size_t)a * cols + c);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i < mm) acc[i] = fmaf(Pl[(m0 + i) * ra + a], b, acc[i]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < mm) out[(size_t)(m0 + i) * cols + c] = acc[i];
        }
    }
}

// 16-byte asynchronous copy global -> shared, past L1
__device__ __forceinline__ void tt_cp_async16(void* smem_dst, const void* gsrc)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}

// ... of the first `floats` of the 16 bytes only (at least one float), the others zero
__device__ __forceinline__ void tt_cp_async16_cut(void* smem_dst, const void* gsrc, uint64_t floats)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gsrc), "r"(floats < 4 ? (unsigned)floats * 4u : 16u) : "memory");
}

// left operand of level k (2..K-1) for node v: P_{k-1} of its parent (k = 2: the slice of the first core)
__device__ __forceinline__ const float* tt_left_operand(const WsView& w, const TableDesc& td, int k, uint32_t v)
{
    if (k == 2) {
        const uint32_t i1 = w.val[2][v] / (uint32_t)td.n[1];
        return td.core[0] + (size_t)i1 * td.slice_floats[0];
    }
    return w.pbuf[k - 1] + (size_t)w.parent[k][v] * w.stride[k - 1];
}

// groups swept in digit-major order (neighbours share the big slice of core K-1, which is then fetched from L2 once per
// run instead of once per group); otherwise in natural order
__host__ __device__ __forceinline__ bool tt_digit_major(const WsView& w) { return w.K >= 3 && !(w.ablation & 1); }

// cost of group g (a level-(K-1) node): FMAs of its intermediate product and of its rows, c_k = P_{k-1} r_{k-1} d_k r_k
__device__ __forceinline__ uint32_t tt_group_cost(const WsView& w, const TableDesc& td, uint32_t g)
{
    const int K = w.K;
    const uint32_t nchild = w.cstart[K - 1][g + 1] - w.cstart[K - 1][g];
    const uint64_t c_last = (uint64_t)td.P[K - 1] * td.r[K - 1] * td.d[K - 1];
    const uint64_t c_mid = K >= 3 ? (uint64_t)td.P[K - 2] * td.r[K - 2] * td.d[K - 2] * td.r[K - 1] : 0;
    return (uint32_t)(((c_mid + (uint64_t)nchild * c_last) >> w.cost_shift) + 1);
}

// group range (K = 2: row range) [g0, g1) of work unit q of table t: an equal-cost slice of the table's level-(K-1) groups in sweep order
// (called by one thread per unit, once per forward: k_partition, k_group_cluster)
__device__ __forceinline__ void tt_unit_range(const WsView& w, int t, int q, uint32_t& g0, uint32_t& g1)
{
    const TableDesc& td = w.tdesc[t];
    const int lvl = w.K - 1;
    if (w.K == 2) {   // ranges of rows, see generic.cuh
        const uint32_t u0 = w.tb[2][t], n = w.tb[2][t + 1] - u0;
        const uint32_t Q = min((uint32_t)td.units, max(1u, n / TT_UNIT_ROWS));
        if ((uint32_t)q >= Q) { g0 = u0; g1 = u0; return; }
        g0 = u0 + (uint32_t)((uint64_t)n * (uint32_t)q / Q);
        g1 = u0 + (uint32_t)((uint64_t)n * (uint32_t)(q + 1) / Q);
        return;
    }
    const uint32_t a = w.tb[lvl][t], b = w.tb[lvl][t + 1];
    // the host sizes the grid for the largest possible number of groups; with fewer groups in this batch the table is
    // cut into fewer units (at least td.unit_groups groups each) and the surplus CTAs leave at once
    int Q = td.units;
    {
        const bool pair = (td.fast == 5 || td.fast == 6 || td.fast == 8 || td.fast == 9) && w.tb[lvl][w.T] >= w.paired_groups;
        const int by_groups = (int)(pair ? (b - a + 2 * TT_UNIT_GROUPS - 1) / (2 * TT_UNIT_GROUPS) : (b - a) / (uint32_t)td.unit_groups);
        if (Q > by_groups) Q = by_groups < 1 ? 1 : by_groups;
        if (td.fast < 0 && (td.d[w.K - 1] & 3) != 0 && w.tb[lvl][w.T] >= 2 * TT_UNIT_GROUPS_ANY * w.few_units) {
            const int by_rows = (int)max((w.tb[w.K][t + 1] - w.tb[w.K][t]) / TT_UNIT_ROWS_ODD, (b - a) / 32u);
            if (Q > by_rows) Q = by_rows < 1 ? 1 : by_rows;
        }
    }
    if (q >= Q) { g0 = a; g1 = a; return; }
    if (w.equal_units) {   // equal group counts
        g0 = a + (uint32_t)((uint64_t)(b - a) * (uint64_t)q / Q);
        g1 = a + (uint32_t)((uint64_t)(b - a) * (uint64_t)(q + 1) / Q);
        return;
    }
    const uint64_t ca = w.cost[a], cb = w.cost[b];
    const uint64_t lo_c = ca + (cb - ca) * (uint64_t)q / Q, hi_c = ca + (cb - ca) * (uint64_t)(q + 1) / Q;
    // first group whose exclusive cost >= target
    auto lower = [&](uint64_t target) {
        uint32_t lo = a, hi = b;
        while (lo < hi) {
            uint32_t mid = lo + ((hi - lo) >> 1);
            if ((uint64_t)w.cost[mid] < target) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    g0 = q == 0 ? a : lower(lo_c);
    g1 = q == Q - 1 ? b : lower(hi_c);
}

// Group range of a sweep's CTA, and how many of its groups a warp takes at a time (up to ng).  FEW: the batch may have few groups; without
// branches, so that the loads of the table's descriptor that follow are issued with these (with them behind a branch 21 tables' backward
// sweep of 14 k groups took 115 us instead of 100).
template <bool FEW>
__device__ __forceinline__ uint2 tt_sweep_unit(const WsView& w, int t, uint32_t ng, uint32_t& step)
{
    step = ng;
    if (!FEW) return w.unit_rng[t * w.units_per_table + blockIdx.x];
    const uint32_t q = blockIdx.y, Q = w.units_per_table, total = w.tb[w.K - 1][w.T], a = w.tb[w.K - 1][t], n = w.tb[w.K - 1][t + 1] - a;
    const uint2 unit = w.unit_rng[t * Q + min(q, Q - 1)];
    const bool few = total < w.few_units * TT_FEW_LIMIT, none = q >= Q;
    const uint32_t per = max(max((uint32_t)TT_FEW_GROUPS, __float2uint_ru((float)total * w.few_share)), __float2uint_ru((float)n * w.cta_share) + 1);
    const uint32_t lo = min(q * per, n), hi = min(lo + per, n);
    if (few) step = min(ng, (per + 3) / 4);
    return make_uint2(few ? a + lo : none ? 0u : unit.x, few ? a + hi : none ? 0u : unit.y);
}

__device__ __forceinline__ int tt_find_table64(const int64_t* __restrict__ tb, int T, int64_t v)
{
    int lo = 0, hi = T;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (tb[mid] <= v) lo = mid; else hi = mid;
    }
    return lo;
}
