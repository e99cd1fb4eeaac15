// Kernel launch interface of the batched column-wise SpGEMM (host side of kernels.cu).
//
// Work is expressed in an "item space": a batch holds nprod products
// C_i = A_i * B_i (descriptors in device memory); item u = item_base_i + p is the
// p-th stored column of B_i and produces one output column (or one DCSC column).
// The flat product is a batch of one; the SUMMA stage products, the stage merge
// and spgemm_batch are larger batches.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace sg {

// Column tiers.  An item's capacity bound is cap = min(flops, m) >= nnz of its output.
//   bin 0                          : cap == 0 (empty output column)
//   bins BIN_SORT0 .. +NSORT-1     : at most 16, 32 .. 1024 products (sort tier, up to
//                                    TierCfg::sort_max products; 16 products always)
//   bins BIN_WARP0 .. +NWARP-1     : warp-wide hash tables of 64 .. 1024 slots (>= 2 cap)
//   bins BIN_BLK0 .. +NBLK-1       : CTA-wide hash tables of 2048 .. 8192 slots (>= 2 cap)
//   bin NBIN-1                     : slab tier (long columns cut into row slabs)
constexpr int NSORT = 7;
constexpr int NWARP = 5;
constexpr int NBLK = 3;
constexpr int NBIN = 1 + NSORT + NWARP + NBLK + 1;
constexpr int BIN_SORT0 = 1;
constexpr int BIN_WARP0 = BIN_SORT0 + NSORT;
constexpr int BIN_BLK0 = BIN_WARP0 + NWARP;
constexpr int BIN_DENSE = NBIN - 1;
// Tier of a bin in the plan's statistics: 0 empty, 1 up to warp_max_flops, 2 up to
// block_max_flops, 3 long columns.  A sort bin holds columns of both kinds: `cap` tells.
__host__ __device__ constexpr int tier_of_bin(int b, int64_t cap, int warp_max) {
    return b == 0 ? 0 : b >= BIN_DENSE ? 3 : b >= BIN_BLK0 || (b > BIN_SORT0 && b < BIN_WARP0 && cap > warp_max) ? 2 : 1;
}
constexpr int TINY_MAX = 16;
constexpr int WARP_TBL0 = 64;
constexpr int BLK_TBL0 = 2048;
// most row slabs of one long column
constexpr int MAX_PARTS = 64;
// default most rows of one slab: its row bitmap (and ranks) then leave room for four CTAs of
// the counting pass per SM and three (up to about 273,000 rows four) of the numeric pass.  R-MAT 20 flat FP64 with
// one column cut at 2^19 / 2^18 / 2^17 rows: counting 31.3 / 25.3 / 32.3 ms, numeric 55.3 /
// 51.2 / 56.2 ms; 300,007 rows are better whole than in two slabs (boolean 2.6 against 3.1 ms)
constexpr int DEFAULT_SLAB_ROWS = 327680;
// default target flops per slab: every slab repeats its binary searches per entry of
// B(:,j) and its bitmap set-up, so larger slabs pay up to about this size (R-MAT
// scale 20 flat: 8192 / 16384 / 32768 / 65536 / 131072 flops per slab give 74.8 /
// 67.9 / 64.5 / 62.3 / 62.1 ms for the FP64 numeric pass)
constexpr int DEFAULT_PART_FLOPS = 65536;

// copies of the analysis counters (bin counts, then total flops), two 128-byte lines each
constexpr int CTR_REP = 16;
constexpr int CTR_STRIDE = 32;
constexpr int CTR_SORT2 = NBIN + 1;   // after the total flops: columns of the sort bins that count as tier 2
static_assert(CTR_SORT2 < CTR_STRIDE, "a copy keeps to its lines");

struct TierCfg {
    int warp_max;     // cap <= warp_max -> warp tables (<= 512)
    int block_max;    // cap <= block_max -> CTA tables (<= 4096)
    int sort_max = 0; // columns of at most this many products (and cap <= block_max) go to the
                      // sort tier: sort_max_products(rows), less where another tier is faster
    int dense_rows;   // RB, most rows of one slab (bitmap bits in shared memory)
    int part_flops;   // target flops per slab of a long column
};

// Everything a pass needs about slab s before its work starts, written by the
// boundary pre-pass (and, for the numeric pass, completed once C's offsets are
// known): the passes copy the next slab's record into shared memory while the
// current slab runs, so a slab starts without a chain of dependent loads.
struct __align__(16) SlabRec {
    int32_t prod, col;   // the long column: product and stored column of B
    int32_t r0, r1;      // rows [r0, r1) of the slab
    int32_t rb;          // output row base of the column
    int32_t cnt;         // rows of the slab's row set (counting pass)
    int64_t bs, be;      // B(:,j) is entries [bs, be)
    int64_t bnd;         // this slab's row of the boundary table in `bnd`
    int64_t u;           // item index of the column
    int64_t ob;          // where the slab's rows start in C (numeric pass)
    int64_t soff;        // where its row set is stored (< 0: none)
    int64_t sab;         // the column's rows P + 1 and P + 2 of `bnd`: where each A(:,k) starts
};
static_assert(sizeof(SlabRec) == 80, "five 16-byte chunks");

// State of the slab tier shared by its kernels.  Slab s = sbase[d] + q is slab q
// of long column d (position d in the dense list); items[s] = (d, q).
struct DenseWork {
    const int2* dlist = nullptr;          // long columns (product, stored column)
    int64_t ndense = 0;
    const int2* items = nullptr;          // slabs (d, q)
    const unsigned long long* nitems = nullptr;   // device count of slabs
    int64_t nslabs = 0;                   // host copy of the count (0 before it is known)
    const int8_t* nparts = nullptr;       // slabs per long column
    const int32_t* sbase = nullptr;       // first slab of each long column
    int32_t* scount = nullptr;            // rows per slab (symbolic pass)
    int32_t* spref = nullptr;             // rows of the column's earlier slabs
    int64_t* soff = nullptr;              // where each slab's row set is stored
    uint32_t* store = nullptr;            // row sets: bitmap words, or rows ascending
    int64_t store_cap = 0;                // entries of store
    unsigned long long* store_ctr = nullptr;
    const int* vals_zero = nullptr;       // boolean semiring: some operand value is false
    int32_t* bnd = nullptr;               // slab boundaries: per long column, P + 3 rows of deg:
                                          // offsets into every A(:,k) (row P: its length),
                                          // then where A(:,k) starts (low, high 32 bits)
    const int64_t* bbase = nullptr;       // where each long column's boundary table starts
    SlabRec* rec = nullptr;               // per slab: its record
    int* err = nullptr;                   // nonzero: a capacity was exceeded
    int RB = 1 << 19;                     // most rows per slab
    bool many_short = false;              // slabs of few entries of B, most columns cut into several
    int kinds = 0;                        // bit 0: some long column's A is read in aligned quads, bit 1: some is not
    // block mode (every A_i has at most BLOCK_TIER_MAX_ROWS rows): long columns
    // are counted with row bitmaps and computed by the block tier; no slabs
    bool dcol = false;
};

// Products whose every A_i has at most this many rows run their numeric pass in
// the block tier (two-level row bitmap per column, L2 reductions; blocktier.cu)
// and count their columns with row bitmaps.
constexpr int BLOCK_TIER_MAX_ROWS = 32768;

// Most products of a column whose 32-bit keys in the sort tier (sorttier.cu) hold its rows:
// a key is the row above log2(products) bits of slot, and all ones marks an empty slot.
// 0: the rows leave no room even for 16 products.
inline int sort_max_products(int64_t max_m) {
    for (int n = 1024, sb = 10; n >= TINY_MAX; n /= 2, --sb)
        if (max_m <= (int64_t(1) << (32 - sb)) - 1) return n;
    return 0;
}

struct Items {
    const Prod* prods = nullptr;        // device, nprod descriptors
    const int64_t* item_base = nullptr; // device, nprod + 1 (prefix of stored columns of B_i)
    int64_t nprod = 0;
    int64_t nitems = 0;
    int64_t total_bnz = 0;              // sum of nnz(B_i): cursor stride per dense part
    int64_t max_m = 0;                  // most rows of any A_i
    // A-column cache (DCSC A only): for every stored entry B_i(k, j), where A_i(:,k)
    // starts and how long it is, filled by the analysis pass so that later passes
    // skip the DCSC lookup.  Indexed by bnz_base + position within B_i.
    int64_t* acs = nullptr;
    int32_t* acl = nullptr;
};

// A(:,k) for the B entry at position t of product pr (cached when the engine has
// the A-column cache, else looked up).
__device__ __forceinline__ void a_col(const Items& it, const Prod* pr, int64_t t, int32_t k, int64_t& s, int64_t& e) {
    if (it.acs) {
        const int64_t i = pr->bnz_base + (t - __ldg(pr->B.cp));
        s = __ldg(it.acs + i);
        e = s + __ldg(it.acl + i);
    } else {
        col_range(pr->A, k, s, e);
    }
}

// CTA-wide hash tables order their numeric output through a shared-memory row
// bitmap (instead of sorting) when every A_i has at most this many rows.
constexpr int64_t BM_MAX_ROWS = 262144;
// The same for warp tables (one bitmap per warp), and only where sorting costs more.
constexpr int64_t BM_WARP_MAX_ROWS = 32768;
constexpr int BM_WARP_MIN_TBL = 256;   // smaller tables hold too few rows to prefer the bitmap

// Side streams and events of a context (created at its first pass of several launches).
struct LanePool {
    static constexpr int NSIDE = 3;
    cudaStream_t side[NSIDE] = {nullptr};
    cudaEvent_t start = nullptr, done[NSIDE] = {nullptr};
    bool ready = false, failed = false;
    bool init();
    void destroy();
};

// The streams that the launches of one pass go to.  The tiers of a pass work on columns of
// their own, so their launches may overlap: they take turns on the context's stream and the
// pool's side streams, which start after everything queued on the context's stream before
// this object and are joined into it when the object goes (a stream capture of the
// context's stream captures the fork and the join with it).  From a plain stream: one lane.
// A pass has up to 16 launches whose last CTAs leave most of the chip idle, 10 to 25 us each
// even for a handful of columns.  Whole calls, one lane against four: BFS step 343 -> 276 us,
// restriction products 2057 -> 1572 us, 20 int64 pairs 1830 -> 1524 us, R-MAT 18 SUMMA FP64
// 26.2 -> 24.7 ms.  The fork and the join cost about 8 us, so a pass of one launch has none.
class Lanes {
  public:
    Lanes(cudaStream_t main) : main_(main) {}
    Lanes(cudaStream_t main, LanePool* pool);   // pool null or unusable: one lane
    ~Lanes();
    Lanes(const Lanes&) = delete;
    Lanes& operator=(const Lanes&) = delete;
    cudaStream_t next() const;

  private:
    cudaStream_t main_;
    LanePool* pool_ = nullptr;
    mutable int turn_ = 0;
    mutable bool used_[LanePool::NSIDE] = {false};
};

// flops and bin per item, product id per item, nnz_item = 0, bin counts and total flops (CTR_REP partial
// copies each, CTR_STRIDE entries apart: bin_count[r * CTR_STRIDE + b]).
// With feat != nullptr also the 8 predictor inputs per item; `sketch` holds the
// per-column row sketches of the A operands concatenated, product i's starting
// at sketch_base[i].
void launch_analyze(cudaStream_t st, const Items& it, TierCfg cfg, int64_t* flops, uint8_t* bin, int32_t* item_prod,
                    unsigned long long* bin_count, unsigned long long* flops_total, const uint64_t* sketch,
                    const int64_t* sketch_base, float* feat, int64_t* maxlen, int64_t* nnz_item);
void launch_row_sketch(cudaStream_t st, const DMat& A, uint64_t* sketch);
// per-bin lists of the items; cnt holds the bins' counts in `rep` copies CTR_STRIDE apart,
// cursor NBIN zeros; off_out gets where every list starts
void launch_bin_scatter(cudaStream_t st, const Items& it, const uint8_t* bin, const int32_t* item_prod,
                        const unsigned long long* cnt, int rep, unsigned long long* cursor, int64_t* off_out,
                        int2* list);
// out = exclusive scan of the exact counts nnz_item (out[nitems] the total), the items' numeric
// bins nbin, the bins' counts cnt[NBIN] and lists; cnt[0, 2 NBIN) is zero before
void launch_count_scan(cudaStream_t st, const Items& it, TierCfg cfg, const uint8_t* bin, const int64_t* flops,
                       const int32_t* item_prod, const int64_t* nnz_item, int64_t* out, void* tmp, uint8_t* nbin,
                       unsigned long long* cnt, int2* list);
// slabs of the long columns (position d in the dense list, slab q); P_d slabs of at
// most RB rows each; *store_bound accumulates the entries their row sets can need, *kinds
// (may be null) the bits of DenseWork::kinds
void launch_dense_items(cudaStream_t st, const Items& it, const int2* dense_list, int64_t ndense,
                        const int64_t* flops, int part_flops, int RB, int2* items, unsigned long long* nitems,
                        int8_t* nparts, int32_t* sbase, unsigned long long* store_bound, int64_t* bbase,
                        unsigned long long* bnd_total, unsigned long long* kinds);
// entries that a slab of at most RB rows can add up in shared memory (0: semirings without)
int slab_acc_entries(int sr, int RB);
// whether A of the product can be read in aligned quads by the slab passes
bool slab_quads(const Prod& pr);
// *flag = 1 when an operand of some product stores a false value (boolean semiring); `most`: the
// entries of the largest operand
void launch_false_values(cudaStream_t st, const Items& it, int64_t most, int* flag);
// *flag = 1 when one of the n bytes at vals is 0 (vals == nullptr: nothing)
void launch_any_false(cudaStream_t st, const void* vals, int64_t n, int* flag);

// which: 1 = hash-table tiers, 2 = long columns (slab tier, or the block tier in block mode), 3 = both
template <class SR>
void launch_symbolic(const Lanes& st, const Items& it, TierCfg cfg, const int2* list, const int64_t* bin_off,
                     const int64_t* bin_cnt, const DenseWork& dw, int64_t* nnz_item, int which = 3);
template <class SR>
void launch_numeric(const Lanes& st, const Items& it, TierCfg cfg, const int2* list, const int64_t* bin_off,
                    const int64_t* bin_cnt, const DenseWork& dw, const int64_t* Coff, int32_t* Cir,
                    typename SR::T* Cv, int which = 3);

// numeric pass of the hash tiers into a predicted layout: cap_off are capacity offsets;
// every item's exact count goes to nnz_item, items that do not fit are not written
template <class SR>
void launch_numeric_predicted(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                              const int64_t* bin_cnt, const DenseWork& dw, const int64_t* cap_off, int64_t* nnz_item,
                              int32_t* Cir, typename SR::T* Cv);

// numeric pass of the block tier (blocktier.cu); with nnz_item the counts are recorded and
// a column is written only when it fits its slots Coff[u+1] - Coff[u]
template <class SR>
void launch_block_tier(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                       const int64_t* bin_cnt, const DenseWork& dw, int64_t* nnz_item, const int64_t* Coff,
                       int32_t* Cir, typename SR::T* Cv, int which);
// numeric pass of the sort bins (sorttier.cu); nnz_item as for launch_block_tier
template <class SR>
void launch_sort_tier(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                      const int64_t* bin_cnt, int64_t* nnz_item, const int64_t* Coff, int32_t* Cir,
                      typename SR::T* Cv, const int* vals_zero);
// counting pass of the sort bins
void launch_sort_count(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                       const int64_t* bin_cnt, int64_t* nnz_item);
// nnz of long columns = sum of their slab counts (and each slab's start in its column)
void launch_sum_parts(cudaStream_t st, const Items& it, const DenseWork& dw, int64_t* nnz_item);
// per-product column pointers from item offsets: out[colbase_i + j] for j in [0, n_i]
void launch_colptrs(cudaStream_t st, const Items& it, const int64_t* colbase, int64_t total_cols, const int64_t* Coff,
                    int64_t* out);
// out[i] = Coff[item_base[i]] for i in [0, np]: where each product's output starts
void launch_gather_offsets(cudaStream_t st, const int64_t* Coff, const int64_t* item_base, int64_t np, int64_t* out);
// out[0] = 0, out[i+1] = sum_{t <= i} in[t]; tmp needs scan_tmp_bytes(n)
size_t scan_tmp_bytes(int64_t n);
void launch_exclusive_scan(cudaStream_t st, const int64_t* in, int64_t n, int64_t* out, void* tmp);
void launch_fill_i64(cudaStream_t st, int64_t* p, int64_t n, int64_t v);
// per-tier totals {cols, flops, nnz(C), nnz(B)} x 4 tiers into out[16] (device, zeroed by caller)
void launch_tier_stats(cudaStream_t st, const Items& it, const uint8_t* bin, const int32_t* item_prod,
                       const int64_t* flops, const int64_t* nnz_item, int warp_max, unsigned long long* out);


// raises a kernel's dynamic shared-memory limit on the current device to at least `bytes`
void smem_at_least(const void* fn, size_t bytes);
// streaming multiprocessors of the current device (queried once per device)
int sm_count();

// process-wide count of kernel launches made by this library
void note_launch(int n = 1);
int64_t launches();

}  // namespace sg
